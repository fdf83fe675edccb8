// Instantiations of the strided-axis passes: float32 register passes.
//
// Lines of 64 points and more run on line_kernel (line_pass.cuh), shorter ones
// on the one-column kernel of yz_kernel.cuh: a thread of line_kernel takes at
// least 8 values of two columns, so a 16-point tile would be half a warp, and on
// 32-point lines its CTAs of 512 threads cost a small grid more than they save
// (32^3 step 44.6 -> 46.1 us).
// Against the kernels they replaced (8 or 16 values per thread, two exchanges
// per transform, three for 1024 points), z_div / z_abs / y of three spectra:
//   512^3   0.991 / 0.663 / 0.565 ms -> 0.657 / 0.468 / 0.555 ms
//   1024^3 11.12  / 6.93  / 5.0  ms -> 6.16  / 4.17  / 4.53 ms
//   256^3   133   / 90    / 76   us -> 89    / 74    / 75   us
// (with the spectra in blocks of columns, kwgb_internal.h).
#include "line_pass.cuh"

namespace kwgb {

template <int L, int OP>
static cudaError_t launch_f32(const YZK& a, int items, cudaStream_t s) {
    // y lines of 1024 points of 8-real rows, in spectra beyond L2: HBM bounds the pass and 3 of
    // a tile's 8 columns are idle, so one-exchange transforms save nothing, and the one-column kernel
    // is faster (step of 1024 x 1024 x 8 1.61 -> 1.58 ms; in L2, 256 x 1024 x 8, 317 -> 348 us)
    if constexpr (L == 10 && OP < 2) {
        if (a.clip == 0 && a.g.nh <= 8) return launch_t<L, OP, 0>(a, items, s);
    }
    if constexpr (L >= 6) return launch_line<L, OP>(a, s);
    else return launch_t<L, OP, 0>(a, items, s);
}

template <int OP>
static cudaError_t by_size(const YZK& a, int logn, int items, cudaStream_t s) {
    switch (logn) {
#define CASE(L) case L: return launch_f32<L, OP>(a, items, s);
        KWGB_LOG_CASES(CASE)
#undef CASE
    }
    return cudaErrorInvalidValue;
}

cudaError_t yz_dispatch_f32(const YZK& a, int op, int logn, int items, cudaStream_t s) {
    switch (op) {
        case OP_Y_FWD: return by_size<OP_Y_FWD>(a, logn, items, s);
        case OP_Y_INV: return by_size<OP_Y_INV>(a, logn, items, s);
        case OP_Z_GRAD_FWD: return by_size<OP_Z_GRAD_FWD>(a, logn, items, s);
        case OP_Z_GRAD_BWD: return by_size<OP_Z_GRAD_BWD>(a, logn, items, s);
        case OP_Z_DIV: return by_size<OP_Z_DIV>(a, logn, items, s);
        case OP_Z_ABS: return by_size<OP_Z_ABS>(a, logn, items, s);
        case OP_Z_DIV_FWD: return by_size<OP_Z_DIV_FWD>(a, logn, items, s);
        case OP_Z_DIV_SUM: return by_size<OP_Z_DIV_SUM>(a, logn, items, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace kwgb
