// Host side of the strided-axis passes: tensor-map encoding and launch
// dispatch (the kernels are in yz_kernel.cuh, instantiated per precision form
// in yz_f32.cu, yz_bf16.cu and yz_f16.cu).
#include "yz_kernel.cuh"

namespace kwgb {

// ---------------------------------------------------------------- host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*,
                                  CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                  CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    }
    return fn;
}

// The last block of a spectrum is never full (nx/2 + 1 columns).  In a spectrum of 64 MB and
// more its tiles come through a tensor map of their own, which ends with the last column and
// promotes no fetch, so that the padding beside it stays in HBM: at 512 x 512 x 128 the forward
// y pass of one spectrum reads 206 MB with the 256-byte pieces, 172 without (136 are needed: the Nyquist column's
// sectors bring their 128-byte lines), at 1024 x 1024 x 128 896 and 730.  Steps: 1024 x 1024 x 128
// 9.06 -> 8.62 ms, 512^3 7.54 -> 7.45, 512 x 1024 x 8 0.81 -> 0.72.  Smaller spectra stay in L2, where the
// padding costs nothing and the clipped map does (512 x 512 x 16, 34 MB, 455 -> 469 us).
// Rows of 8 reals (5 columns of 16, next to one another) keep the promotion: it brings the rows
// that the next tiles take (step of 1024 x 1024 x 8 1.64 -> 1.61 ms; rows of 16 reals lose 2 %).
static bool clips_last_block(const GridC& g) { return spec_elems(g) * sizeof(float2) >= (size_t)64 << 20; }

// map[0]: every block at its full width; map[1]: the last one up to the last column
template <int LOGN, bool ISY, int MIXED>
static int encode_box(const GridC& g, float2* ptr, CUtensorMap (&map)[2]) {
    using Sh = TShape<LOGN, ISY, MIXED>;
    EncodeTiledFn fn = encode_fn();
    if (!fn) return -1;
    // a tile's CX columns lie in one block (CX divides the block width, 16 or 32)
    static_assert(16 % Sh::CX == 0, "tile width");
    const cuuint64_t w = (cuuint64_t)1 << g.lb, row = w * 8, full = (g.nh - 1) / w;
    const cuuint64_t strides[3] = {row, g.ny * row, (cuuint64_t)g.ny * g.nz * row};
    const cuuint32_t box[4] = {(cuuint32_t)Sh::CX, ISY ? (cuuint32_t)Sh::BOX : 1u, ISY ? 1u : (cuuint32_t)Sh::BOX, 1u};
    const cuuint32_t es[4] = {1, 1, 1, 1};
    for (int last = 0; last < 2; ++last) {
        const cuuint64_t dims[4] = {last ? g.nh - full * w : w, (cuuint64_t)g.ny, (cuuint64_t)g.nz, last ? 1 : full + 1};
        const CUresult r = fn(&map[last], CU_TENSOR_MAP_DATA_TYPE_INT64, 4, ptr + (last ? full * spec_block(g) : 0), dims,
                              strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                              last && g.nh > 8 ? CU_TENSOR_MAP_L2_PROMOTION_NONE : CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r != CUDA_SUCCESS) return -2;
    }
    return 0;
}


int make_spec_maps(const GridC& g, float2* ptr, SpecBuf* out) {
    out->p = ptr;
    int e = -3;
    switch (g.logny) {
#define CASE(L) case L: e = g.mixed ? encode_box<L, true, 1>(g, ptr, out->ymap) : encode_box<L, true, 0>(g, ptr, out->ymap); break;
        KWGB_LOG_CASES(CASE)
#undef CASE
    }
    if (e) return e;
    switch (g.lognz) {
#define CASE(L) case L: e = g.mixed ? encode_box<L, false, 1>(g, ptr, out->zmap) : encode_box<L, false, 0>(g, ptr, out->zmap); break;
        KWGB_LOG_CASES(CASE)
#undef CASE
    }
    return e;
}

static cudaError_t launch_op(int op, const YZK& a, int logn, int items, cudaStream_t s) {
    if (a.g.mixed == 2) return yz_dispatch_f16(a, op, logn, items, s);
    if (a.g.mixed == 1) return yz_dispatch_bf16(a, op, logn, items, s);
    return yz_dispatch_f32(a, op, logn, items, s);
}

static void set_maps(YZK& a, int i, const CUtensorMap (&m)[2]) {
    a.map[i] = m[0];
    a.map[3 + i] = m[1];
}

static int chunk_count(int nh, int cx) { return (nh + cx - 1) / cx; }

// tile width of the pass (the tensor-core forms share one shape)
template <bool ISY>
static int cx_of(int logn, int mixed) {
    switch (logn) {
#define CASE(L) case L: return mixed ? TShape<L, ISY, 1>::CX : TShape<L, ISY, 0>::CX;
        KWGB_LOG_CASES(CASE)
#undef CASE
    }
    return 16;
}

cudaError_t launch_y_pass(const GridC& g, int dir, const SpecBuf* const* in, float2* const* out,
                          int ncomp, int* flag, cudaStream_t s) {
    YZK a;
    memset(&a, 0, sizeof(a));
    a.g = g;
    for (int i = 0; i < ncomp; ++i) {
        set_maps(a, i, in[i]->ymap);
        a.out[i] = out[i];
    }
    a.ncomp = ncomp;
    a.nloads = 1;
    a.flag = flag;
    a.clip = clips_last_block(g) ? (g.nh - 1) >> g.lb : -1;
    const int items = chunk_count(g.nh, cx_of<true>(g.logny, g.mixed)) * g.nz * ncomp;
    return launch_op(dir < 0 ? OP_Y_FWD : OP_Y_INV, a, g.logny, items, s);
}

cudaError_t launch_z_op(const GridC& g, int kind, const SpecBuf* const* in, float2* const* out, int* flag,
                        cudaStream_t s) {
    YZK a;
    memset(&a, 0, sizeof(a));
    a.g = g;
    a.flag = flag;
    a.clip = clips_last_block(g) ? (g.nh - 1) >> g.lb : -1;
    for (int i = 0; i < 3; ++i) a.out[i] = out[i];
    a.short_kappa = g.hk2 <= 1.9999f * g.inv_kmax2;   // with room for the rounding of k^2
    if (kind == Z_GRAD_FWD || kind == Z_GRAD_BWD) {
        set_maps(a, 0, in[0]->zmap);
        a.nloads = 1;
        a.load_comp[0] = 0;
    } else if (kind == Z_DIV || kind == Z_DIV_FWD || kind == Z_DIV_SUM) {
        for (int i = 0; i < 3; ++i) {
            set_maps(a, i, in[i]->zmap);
            a.load_comp[i] = i;
        }
        a.nloads = 3;
    } else {
        int n = 0;
        for (int t = 0; t < 2; ++t)
            if (in[t]) {
                set_maps(a, t, in[t]->zmap);
                a.load_comp[n++] = t;
            }
        a.nloads = n;
        if (n == 0) return cudaSuccess;
    }
    const int items = chunk_count(g.nh, cx_of<false>(g.lognz, g.mixed)) * g.ny;
    switch (kind) {
        case Z_GRAD_FWD: return launch_op(OP_Z_GRAD_FWD, a, g.lognz, items, s);
        case Z_GRAD_BWD: return launch_op(OP_Z_GRAD_BWD, a, g.lognz, items, s);
        case Z_DIV: return launch_op(OP_Z_DIV, a, g.lognz, items, s);
        case Z_DIV_FWD: return launch_op(OP_Z_DIV_FWD, a, g.lognz, items, s);
        case Z_DIV_SUM: return launch_op(OP_Z_DIV_SUM, a, g.lognz, items, s);
        case Z_ABS: return launch_op(OP_Z_ABS, a, g.lognz, items, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace kwgb
