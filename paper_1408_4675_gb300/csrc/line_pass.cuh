#pragma once
// Float32 y and z passes of lines of 64 to 1024 points: one shared-memory
// exchange per transform, packed arithmetic.
//
// A pass over a tile (CX columns x one whole line) is bound by the SM, not by
// HBM: issue slots, and the shared-memory/L1 data path.  With 8 values per
// thread a 512-point transform crosses shared memory twice and loads 14
// twiddles per 8 values.  Here a thread holds 32 (or 16 x 2) complex values in
// 64 registers, so that N = 32 x (N / 32) is two register passes with ONE
// exchange between them, in the buffer the TMA tile arrived in, and the
// registers hold PAIRS of values, so that every butterfly of both is one
// packed instruction (pair_fft.cuh):
//   N = 64, 128       (PairLine): two adjacent columns of a line
//   N = 256 to 1024   (HalfLine): two elements of one column
// A pair that is not what memory holds costs register moves.  HalfLine has
// none of them where it counts: the forward transform begins, and the inverse
// transform ends, with the one radix-2 step that runs within the pairs, in
// scalar arithmetic, so its operands and results are single elements; between
// the two, the exchanges carry whole pairs (16 bytes; below 1024 points).
// One CTA of 16 warps (128 registers a thread) runs per SM, as 2 to 8 groups that
// take tiles in turn out of a ring of half as many buffers more, so that loads
// are always under way while every group computes.  A CTA's tiles are
// consecutive ones, so that the 64- or 128-byte rows in its ring are neighbours
// in memory (all tiles dealt out one by one: y 1024^3 4.96 -> 7.9 ms, z_div 512^3 0.74 ->
// 0.84 ms).  The tables come from shared memory: beside the ring the L1 cache
// is too small for them (z_abs 512^3 0.71 ms).
#include "pair_fft.cuh"
#include "yz_kernel.cuh"

namespace kwgb {

// The two line types have the same members.  SWAP: the roles of re and im are
// exchanged, which turns the forward transform into the inverse one.
//   fwd(): tile in shared memory -> transform, slot m of the thread holding
//          elements e0(j, m) and e1(j, m) of columns col0 and col1; the
//          buffer has been read when it returns, but not by every thread yet
//   inv(): the reverse: slots -> transform; the caller gets the outputs one
//          slot at a time (emit(element, first value, second value))

// Two adjacent columns (2 c, 2 c + 1) of a tile: slot m holds element j + TL m of both.
template <int LOGN, int CX_>
struct PairLine {
    static constexpr int N = 1 << LOGN, CX = CX_;
    static constexpr int E = LOGN == 6 ? 8 : 16;
    static constexpr int H = E;                       // pair slots per thread
    static constexpr int TL = N / E, R2 = N / E, NB = E / R2;
    static constexpr int TC = CX / 2;                 // threads across the tile
    static constexpr int THREADS = TC * TL;
    static constexpr int BUF = N * CX;                // complex per buffer
    static constexpr int TW0 = stw_off(N, E);         // the twiddles: start and number of entries (transform, both transforms)
    static constexpr int NTW = (E - 1) * (N / E), NTW2 = NTW;
    __device__ __forceinline__ static int e0(int j, int m) { return j + TL * m; }
    __device__ __forceinline__ static int e1(int j, int m) { return j + TL * m; }
    __device__ __forceinline__ static int col0(int c) { return 2 * c; }
    __device__ __forceinline__ static int col1(int c) { return 2 * c + 1; }

    // transform of values in registers (element j + TL m in slot m), through buf
    template <class Sync>
    __device__ __forceinline__ static void dft(float2 (&re)[H], float2 (&im)[H], float2* buf, int c, int j,
                                               const float2* tw, Sync&& sync) {
        dft_pair<E>(re, im);
#pragma unroll
        for (int r = 1; r < E; ++r) {                 // output r of butterfly j carries w_N^{j r}
            const float2 w = tw[(r - 1) * (N / E) + j];
            cmul2(re[r], im[r], dup2(w.x), dup2(w.y));
        }
        float4* b4 = reinterpret_cast<float4*>(buf) + c;
        sync();                              // the buffer's previous contents have been read
#pragma unroll
        for (int r = 0; r < E; ++r) b4[(j * E + r) * TC] = make_float4(re[r].x, re[r].y, im[r].x, im[r].y);
        sync();
#pragma unroll
        for (int m = 0; m < E; ++m) {
            const float4 t = b4[(j + TL * m) * TC];
            re[m] = make_float2(t.x, t.y);
            im[m] = make_float2(t.z, t.w);
        }
    }
    __device__ __forceinline__ static void end(float2 (&re)[H], float2 (&im)[H]) {
#pragma unroll
        for (int i = 0; i < NB; ++i) {                // butterfly b = j + TL i: slots i + NB r
            float2 a[R2], b[R2];
#pragma unroll
            for (int r = 0; r < R2; ++r) { a[r] = re[i + NB * r]; b[r] = im[i + NB * r]; }
            dft_pair<R2>(a, b);
#pragma unroll
            for (int r = 0; r < R2; ++r) { re[i + NB * r] = a[r]; im[i + NB * r] = b[r]; }
        }
    }
    template <bool SWAP, class Sync>
    __device__ __forceinline__ static void fwd(float2 (&re)[H], float2 (&im)[H], float2* buf, int c, int j,
                                               const float2* tw, Sync&& sync) {
#pragma unroll
        for (int m = 0; m < H; ++m) {
            const float4 t = reinterpret_cast<const float4*>(buf)[(j + TL * m) * TC + c];
            re[m] = make_float2(t.x, t.z);
            im[m] = make_float2(t.y, t.w);
        }
        if constexpr (SWAP) dft(im, re, buf, c, j, tw, sync);
        else dft(re, im, buf, c, j, tw, sync);
    }
    template <bool SWAP>
    __device__ __forceinline__ static void fwd_end(float2 (&re)[H], float2 (&im)[H]) {
        if constexpr (SWAP) end(im, re);
        else end(re, im);
    }
    template <class Sync>
    __device__ __forceinline__ static void inv(float2 (&re)[H], float2 (&im)[H], float2* buf, int c, int j,
                                               const float2* tw, Sync&& sync) {
        dft(im, re, buf, c, j, tw, sync);
    }
    template <class Emit>
    __device__ __forceinline__ static void inv_end(float2 (&re)[H], float2 (&im)[H], int j, Emit&& emit) {
        end(im, re);
#pragma unroll
        for (int m = 0; m < H; ++m) emit(j + TL * m, 0, make_float2(re[m].x, im[m].x), make_float2(re[m].y, im[m].y));
    }
    // a slot's values a (p: element e0, column col0) and b
    __device__ __forceinline__ static void store(float2* p, size_t, float2 a, float2 b, bool v0, bool v1) {
        if (v1) __stcs(reinterpret_cast<float4*>(p), make_float4(a.x, a.y, b.x, b.y));
        else if (v0) __stcs(p, a);
    }
};

// (re, im) * exp(-2 pi i m / 32) in scalar arithmetic
__device__ __forceinline__ float2 rot32(float2 d, int m) {
    if (m == 0) return d;
    if (m == 8) return make_float2(d.y, -d.x);
    const float c = cos32(m), s = -sin32(m);
    if (m > 4 && m < 12) return make_float2(fmaf(-d.y, s, d.x * c), fmaf(d.x, s, d.y * c));   // (the order: cmul2_flat)
    return make_float2(fmaf(d.x, c, -d.y * s), fmaf(d.y, c, d.x * s));
}

// 32 elements of one column, N = 32 TL.  Forward: 32-point butterflies over the
// elements j + TL m, then TL-point ones; inverse: TL-point, then 32-point.
// TL < 32: between them the thread holds P = 16 / TL groups of TL slots, slot
// (p, q) the elements b + 32 q and b + 1 + 32 q with b = 2 (j P + p).
template <int LOGN, int CX_>
struct HalfLine {
    static constexpr int N = 1 << LOGN, CX = CX_;
    static constexpr int H = 16;
    static constexpr int TL = N / 32;
    static constexpr bool WIDE = LOGN == 10;
    static constexpr int P = WIDE ? 1 : 16 / TL;
    static constexpr int TC = CX;
    static constexpr int THREADS = TC * TL;
    static constexpr int BUF = WIDE ? 32 * 33 * CX : N * CX;   // 1024 points: one row of padding after every 32
    static constexpr int TW0 = twh_off(LOGN);         // the twiddles: start, entries of the forward, of both transforms
    static constexpr int NTW = 32 * TL, NTW2 = NTW + 32 * TL;
    __device__ __forceinline__ static int e0(int j, int m) { return WIDE ? j + 64 * m : 2 * (j * P + m / TL) + 32 * (m % TL); }
    __device__ __forceinline__ static int e1(int j, int m) { return WIDE ? j + 64 * m + 32 : e0(j, m) + 1; }
    __device__ __forceinline__ static int col0(int c) { return c; }
    __device__ __forceinline__ static int col1(int c) { return c; }

    template <bool SWAP>
    __device__ __forceinline__ static float2 sw(float2 a) { return SWAP ? make_float2(a.y, a.x) : a; }

    // radix-2 step of elements a, b (inputs m and m + 16 of a 32-point butterfly) into slot m
    __device__ __forceinline__ static void split(float2 a, float2 b, int m, float2& x, float2& y) {
        const float2 s = cadd(a, b), d = rot32(csub(a, b), m);
        x = make_float2(s.x, d.x);
        y = make_float2(s.y, d.y);
    }
    template <bool SWAP, class Sync>
    __device__ __forceinline__ static void fwd(float2 (&re)[H], float2 (&im)[H], float2* buf, int c, int j,
                                               const float2* tw, Sync&& sync) {
        auto run = [&](float2 (&x)[H], float2 (&y)[H]) {
#pragma unroll
            for (int m = 0; m < H; ++m)
                split(sw<SWAP>(buf[(j + TL * m) * CX + c]), sw<SWAP>(buf[(j + TL * (m + 16)) * CX + c]), m, x[m], y[m]);
            dft_pair<H>(x, y);                        // slot u: outputs 2u, 2u + 1
#pragma unroll
            for (int u = 0; u < H; ++u) {
                const float4 t = reinterpret_cast<const float4*>(tw)[u * TL + j];
                cmul2(x[u], y[u], make_float2(t.x, t.y), make_float2(t.z, t.w));
            }
            sync();                          // the tile has been read
            if constexpr (WIDE) {
                float2* b = buf + j * 33 * CX + c;
#pragma unroll
                for (int u = 0; u < H; ++u) {
                    b[2 * u * CX] = make_float2(x[u].x, y[u].x);
                    b[(2 * u + 1) * CX] = make_float2(x[u].y, y[u].y);
                }
                sync();
                const float2* r = buf + j * CX + c;
#pragma unroll
                for (int m = 0; m < H; ++m) split(r[m * 33 * CX], r[(m + 16) * 33 * CX], m, x[m], y[m]);
            } else {
                float4* b = reinterpret_cast<float4*>(buf) + c;
#pragma unroll
                for (int u = 0; u < H; ++u) b[(j * H + u) * CX] = make_float4(x[u].x, x[u].y, y[u].x, y[u].y);
                sync();
#pragma unroll
                for (int m = 0; m < H; ++m) {
                    const float4 t = b[((m % TL) * H + j * P + m / TL) * CX];
                    x[m] = make_float2(t.x, t.y);
                    y[m] = make_float2(t.z, t.w);
                }
            }
        };
        if constexpr (SWAP) run(im, re);
        else run(re, im);
    }
    __device__ __forceinline__ static void groups(float2 (&x)[H], float2 (&y)[H]) {
#pragma unroll
        for (int p = 0; p < P; ++p) dft_pair<H / P>(x + p * (H / P), y + p * (H / P));
    }
    template <bool SWAP>
    __device__ __forceinline__ static void fwd_end(float2 (&re)[H], float2 (&im)[H]) {
        if constexpr (SWAP) groups(im, re);
        else groups(re, im);
    }
    template <class Sync>
    __device__ __forceinline__ static void inv(float2 (&re)[H], float2 (&im)[H], float2* buf, int c, int j,
                                               const float2* tw, Sync&& sync) {
        float2 (&x)[H] = im;
        float2 (&y)[H] = re;
        groups(x, y);                                 // WIDE: even inputs in .x, odd inputs in .y
        if constexpr (WIDE) {
            const float2* w = tw + 32 * TL + j;
#pragma unroll
            for (int k = 0; k < H; ++k) {             // join: outputs k and k + 16 of the 32-point butterfly, w_N^{j r}
                const float2 e = make_float2(x[k].x, y[k].x), o = rot32(make_float2(x[k].y, y[k].y), k);
                const float2 a = cmul(cadd(e, o), w[32 * k]), b = cmul(csub(e, o), w[32 * (k + 16)]);
                x[k] = a;                             // x, y: the two elements themselves until they are written
                y[k] = b;
            }
            sync();
            float2* b = buf + j * 33 * CX + c;
#pragma unroll
            for (int k = 0; k < H; ++k) {
                b[k * CX] = x[k];
                b[(k + 16) * CX] = y[k];
            }
            sync();
            const float2* r = buf + j * CX + c;
#pragma unroll
            for (int u = 0; u < H; ++u) {
                const float2 a0 = r[2 * u * 33 * CX], a1 = r[(2 * u + 1) * 33 * CX];
                x[u] = make_float2(a0.x, a1.x);
                y[u] = make_float2(a0.y, a1.y);
            }
        } else {
            const float4* w = reinterpret_cast<const float4*>(tw) + 16 * TL + j * P;
#pragma unroll
            for (int m = 0; m < H; ++m) {             // slot (p, r): outputs r of butterflies b, b + 1
                const float4 t = w[16 * (m % TL) + m / TL];
                cmul2(x[m], y[m], make_float2(t.x, t.y), make_float2(t.z, t.w));
            }
            float4* b = reinterpret_cast<float4*>(buf) + c;
            sync();
#pragma unroll
            for (int m = 0; m < H; ++m)
                b[((m % TL) * H + j * P + m / TL) * CX] = make_float4(x[m].x, x[m].y, y[m].x, y[m].y);
            sync();
#pragma unroll
            for (int u = 0; u < H; ++u) {
                const float4 t = b[(j * H + u) * CX];
                x[u] = make_float2(t.x, t.y);
                y[u] = make_float2(t.z, t.w);
            }
        }
    }
    template <class Emit>
    __device__ __forceinline__ static void inv_end(float2 (&re)[H], float2 (&im)[H], int j, Emit&& emit) {
        dft_pair<H>(im, re);
#pragma unroll
        for (int k = 0; k < H; ++k) {                 // outputs k, k + 16 (im holds the real role: swap back)
            const float2 e = make_float2(im[k].x, re[k].x), o = rot32(make_float2(im[k].y, re[k].y), k);
            emit(j + TL * k, j + TL * (k + 16), make_float2(e.y + o.y, e.x + o.x), make_float2(e.y - o.y, e.x - o.x));
        }
    }
    // a (element e0) at p, b (element e1) at p + step
    __device__ __forceinline__ static void store(float2* p, size_t step, float2 a, float2 b, bool v0, bool) {
        if (v0) {
            __stcs(p, a);
            __stcs(p + step, b);
        }
    }
};

// One CTA per SM: GR groups of THREADS threads (16 warps together, 128
// registers a thread) take the CTA's tiles in turn out of one ring of NBUF
// tile buffers.
template <int LOGN, bool ISY>
struct LShape {
    using Sh = TShape<LOGN, ISY>;
    using Line = std::conditional_t<(LOGN >= 8), HalfLine<LOGN, Sh::CX>, PairLine<LOGN, Sh::CX>>;
    static constexpr int THREADS = Line::THREADS;
    static constexpr int GR = 512 / THREADS;
    static constexpr int NBUF = GR + GR / 2;
    static constexpr int NTAB = ISY ? Line::NTW : Line::NTW2 + (1 << LOGN) + (1 << LOGN) / 2;   // twiddles, dfz, kz (float2)
    static constexpr int SMEM = (NBUF * Line::BUF + NTAB) * (int)sizeof(float2) + 2 * NBUF * 8;
    static_assert(SMEM <= 227 * 1024 && GR <= 8, "ring too large");
    static_assert(GR * 3 == NBUF * 2, "the barrier rule of the ring (line_kernel)");
};

// exp2 of the operator exponents e log2(k^2 / k_max^2), |e| < 1: the hardware function without the
// handling of denormal results, the same as exp2f there (compared for every float k^2 / k_max^2 in [2^-40, 4)).
// The logarithm is log2f: lg2.approx differs from it in a third of those arguments, by up to
// a unit in the last place more, which the powers multiply (error of k^{y-2} at 256^3 2.7e-7 -> 3.5e-7;
// z_abs would take 0.445 ms at 512^3 instead of 0.468, the eta operator of 256^3 117 us instead of 124).
__device__ __forceinline__ float ex2_normal(float x) {
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// sinc_sq of two values no larger than 2 (the short series, packed).
__device__ __forceinline__ float2 sinc_short2(float2 x2) {
    float2 p = dup2(-1.0f / 39916800.0f);
    p = fma2(p, x2, dup2(1.0f / 362880.0f));
    p = fma2(p, x2, dup2(-1.0f / 5040.0f));
    p = fma2(p, x2, dup2(1.0f / 120.0f));
    p = fma2(p, x2, dup2(-1.0f / 6.0f));
    return fma2(p, x2, dup2(1.0f));
}
// Any argument; out of line, since its long branches would be repeated for every slot.
static __device__ __noinline__ float2 sinc_any2(float2 x2) { return make_float2(sinc_sq(x2.x), sinc_sq(x2.y)); }

// A warp's 32 x 4 H registers in tensor memory: the gradient and the summing
// pass keep one set of values aside there while they transform another (the
// shared memory is taken by the tile ring).
template <int H>
__device__ __forceinline__ void stash_put(uint32_t taddr, const float2 (&re)[H], const float2 (&im)[H]) {
#pragma unroll
    for (int m = 0; m < H; m += 8) {
        uint32_t r[32];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            r[4 * i] = __float_as_uint(re[m + i].x);
            r[4 * i + 1] = __float_as_uint(re[m + i].y);
            r[4 * i + 2] = __float_as_uint(im[m + i].x);
            r[4 * i + 3] = __float_as_uint(im[m + i].y);
        }
        asm volatile(
            "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,"
            "%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};" ::"r"(taddr + 4 * m),
            "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
            "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]),
            "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]),
            "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
            : "memory");
    }
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}
template <int H>
__device__ __forceinline__ void stash_get(uint32_t taddr, float2 (&re)[H], float2 (&im)[H]) {
#pragma unroll
    for (int m = 0; m < H; m += 8) {
        uint32_t r[32];
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
            "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n\ttcgen05.wait::ld.sync.aligned;"
            : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
              "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
              "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
              "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
            : "r"(taddr + 4 * m)
            : "memory");
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            re[m + i] = make_float2(__uint_as_float(r[4 * i]), __uint_as_float(r[4 * i + 1]));
            im[m + i] = make_float2(__uint_as_float(r[4 * i + 2]), __uint_as_float(r[4 * i + 3]));
        }
    }
}

// Tiles: y passes (component, z line, chunk); GRAD (y line, chunk), two
// inverse transforms; DIV and ABS (component, y line, chunk); DIV_SUM (y line,
// chunk), three loads in turn, summed.  Load t of a CTA lands in buffer t mod
// NBUF and is handled by group t mod GR (DIV_SUM: the three loads of a tile by
// one group); the group that has read load t's buffer for the last time issues
// load t + NBUF into it.
// A group whose wait runs out takes no more tiles.  Groups that it would have fed run
// out in turn, and before the CTA exits every load that was issued and not waited for gets one more
// bounded wait: the TMA must not write into shared memory that is no longer the CTA's.
template <int LOGN, int OP>
__global__ void __launch_bounds__(512, 1) line_kernel(const __grid_constant__ YZK a) {
    constexpr bool ISY = OP < 2;
    using Ls = LShape<LOGN, ISY>;
    using Sh = TShape<LOGN, ISY>;
    using Line = typename Ls::Line;
    constexpr int H = Line::H, CX = Sh::CX, TC = Line::TC, THREADS = Line::THREADS, GR = Ls::GR, NBUF = Ls::NBUF;
    constexpr bool GRAD = OP == OP_Z_GRAD_FWD || OP == OP_Z_GRAD_BWD;
    constexpr bool SUM = OP == OP_Z_DIV_SUM;
    constexpr bool STASH = GRAD || SUM;
    constexpr bool BWD = OP == OP_Z_GRAD_BWD || OP == OP_Z_DIV || SUM;    // e^{-ikd/2}: the real part of the operator negated
    extern __shared__ __align__(128) float2 smem[];
    __shared__ int stop[GR];                                  // the load at which a group gave up, or -1
    __shared__ uint32_t tslot;
    // the tables that every thread reads for every value: from shared memory, since
    // the ring leaves the L1 cache too small to keep them
    float2* const tw = smem + NBUF * Line::BUF;
    float2* const dfz = tw + Line::NTW2;
    float* const kz_ = reinterpret_cast<float*>(dfz + (1 << LOGN));
    uint64_t* bar = reinterpret_cast<uint64_t*>(tw + Ls::NTAB);
    const GridC& g = a.g;
    const int grp = threadIdx.x / THREADS, tid = threadIdx.x % THREADS;
    const int c = tid % TC, j = tid / TC;
    const int nchunk = (g.nh + CX - 1) / CX;
    const int lines = ISY ? g.nz : g.ny;
    const int nt = nchunk * lines;                            // tiles of one component
    constexpr int PER = SUM ? 3 : 1;                          // loads per unit of work
    const int units = nt * (ISY ? a.ncomp : (STASH ? 1 : a.nloads));
    // Consecutive units, so that the tiles in a CTA's ring are neighbours in memory; with one
    // tile to a line (rows of 8 or 16 reals) dealt out one by one, so that the tiles of all
    // CTAs are (steps of 1024 x 1024 x 8 1.68 -> 1.64 ms, 512 x 512 x 8 308 -> 304 us).
    const bool one = nchunk == 1;
    const int u0 = one ? (int)blockIdx.x : (int)((int64_t)units * blockIdx.x / gridDim.x);
    const int my = one ? (units - 1 - (int)blockIdx.x) / (int)gridDim.x + 1
                       : (int)((int64_t)units * (blockIdx.x + 1) / gridDim.x) - u0;
    const int us = one ? (int)gridDim.x : 1;
    const int Q = my * PER;
    auto sync = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(1 + grp), "n"(THREADS) : "memory"); };

    if (STASH && threadIdx.x < 32) tc5_alloc(&tslot, 256);
    if (threadIdx.x == 0) {
#pragma unroll
        for (int i = 0; i < 2 * NBUF; ++i) mbar_init(&bar[i], 1);
        fence_mbar_init();
    }
    if (tid == 0) stop[grp] = -1;
    for (int i = threadIdx.x; i < (ISY ? Line::NTW : Line::NTW2); i += 512) tw[i] = __ldg(g.t.tw + Line::TW0 + i);
    if (!ISY)
        for (int i = threadIdx.x; i < (1 << LOGN); i += 512) {
            dfz[i] = __ldg(g.t.dfz + i);
            kz_[i] = __ldg(g.t.kz + i);
        }
    if (STASH) tc5_fence_before();
    __syncthreads();
    uint32_t taddr = 0;                                       // the warp's 64 columns of its 32 lanes
    if (STASH) {
        tc5_fence_after();
        const uint32_t w = threadIdx.x / 32;
        taddr = tslot + ((w % 4) << 21) + (w / 4) * 64;
    }

    auto place = [&](int q, int& chunk, int& line, int& l) {
        int u = u0 + q / PER * us;
        if (SUM) l = q % PER;
        else {
            l = u / nt;
            u -= l * nt;
        }
        line = u / nchunk;
        chunk = u - line * nchunk;
    };
    auto issue = [&](int q) {                 // one thread
        int chunk, line, l;
        place(q, chunk, line, l);
        const int mi = ISY ? l : (l == 0 ? a.load_comp[0] : (l == 1 ? a.load_comp[1] : a.load_comp[2]));
        float2* dst = smem + (q % NBUF) * Line::BUF;
        uint64_t* b = &bar[q % (2 * NBUF)];
        fence_proxy_async_smem();
        mbar_arrive_expect_tx(b, Sh::STAGE * (uint32_t)sizeof(float2) + g.wait_fault_tx);
        int w;
        const CUtensorMap* map = tile_map<true>(a, mi, (chunk * CX) >> g.lb, w);
#pragma unroll
        for (int k = 0; k < Sh::NBOX; ++k) {
            const int x = (chunk * CX) & ((1 << g.lb) - 1);
            if (ISY) tma_load_4d(dst + k * Sh::BOX * CX, map, x, k * Sh::BOX, line, w, b);
            else tma_load_4d(dst + k * Sh::BOX * CX, map, x, line, k * Sh::BOX, w, b);
        }
    };
    after_previous();
    if (threadIdx.x == 0)
        for (int q = 0; q < NBUF && q < Q; ++q) issue(q);
    bool gave_up = false;
    for (int i = grp; i < my; i += GR) {
    for (int q = i * PER; q < (i + 1) * PER; ++q) {
        int chunk, line, l;
        place(q, chunk, line, l);
        float2* buf = smem + (q % NBUF) * Line::BUF;
        const int ca = chunk * CX + Line::col0(c), cb = chunk * CX + Line::col1(c);
        const bool v0 = ca < g.nh, v1 = cb < g.nh;
        // the tile's wavenumbers and its shift operators i k e^{+-ikd/2} along x and y: under way during the wait
        float2 kxy = dup2(0.f), xa = dup2(0.f), xb = dup2(0.f), ya = dup2(0.f);
        if constexpr (!ISY) {
            const float2 kx = make_float2(v0 ? __ldg(g.t.kx + ca) : 0.f, v1 ? __ldg(g.t.kx + cb) : 0.f);
            const float ky = __ldg(g.t.ky + line);
            if (OP != OP_Z_ABS) {
                if (v0) xa = __ldg(g.t.dfx + ca);
                if (v1) xb = __ldg(g.t.dfx + cb);
                ya = __ldg(g.t.dfy + line);
                if (BWD) {
                    xa.x = -xa.x;
                    xb.x = -xb.x;
                    ya.x = -ya.x;
                }
            }
            kxy = fma2(kx, kx, dup2(ky * ky));
        }
        // A wait names a phase by its parity only, so a barrier must not be waited on before its
        // previous phase is known to be over.  Load q has barrier q mod 2 NBUF: the load before
        // on it (q - 2 NBUF) was this group's own, since GR divides 2 NBUF.
        const bool ok = mbar_wait_bounded(&bar[q % (2 * NBUF)], (q / (2 * NBUF)) & 1, a.flag);
        if (!ok) stop[grp] = q;
        float2 re[H], im[H];
        // the buffer is free for its next load once every thread of the group has read it
        auto next = [&]() {
            sync();
            if (tid == 0 && q + NBUF < Q) issue(q + NBUF);
        };
        Line::template fwd<OP == OP_Y_INV>(re, im, buf, c, j, tw, sync);
        if (stop[grp] >= 0) {                         // set before fwd's barriers, so the same for the whole group
            gave_up = true;
            i = my;                                   // no more tiles for this group
            break;
        }
        if constexpr (ISY) {
            next();
            Line::template fwd_end<OP == OP_Y_INV>(re, im);
            float2* out = out_ptr(a, l) + spec_off(g, ca, 0, line);
#pragma unroll
            for (int m = 0; m < H; ++m)
                Line::store(out + ((size_t)Line::e0(j, m) << g.lb), (size_t)(Line::e1(j, m) - Line::e0(j, m)) << g.lb,
                            make_float2(re[m].x, im[m].x), make_float2(re[m].y, im[m].y), v0, v1);
        } else {
            Line::template fwd_end<false>(re, im);
            const size_t es = (size_t)g.ny << g.lb;
            const size_t off = spec_off(g, ca, line, 0);
            const int comp = (OP == OP_Z_ABS && a.load_comp[0] == 1) ? 1 : l;
            auto dz = [&](int m, float2& zr, float2& zi) {
                const float2 za = dfz[Line::e0(j, m)], zb = dfz[Line::e1(j, m)];
                zr = BWD ? make_float2(-za.x, -zb.x) : make_float2(za.x, zb.x);
                zi = make_float2(za.y, zb.y);
            };
            // ZD: the operator includes the shift along z (its own loop, so that the others carry no branch)
            auto apply = [&](auto zd) {
                constexpr bool ZD = decltype(zd)::value;
                const float2 er = comp == 0 ? make_float2(xa.x, xb.x) : dup2(ya.x);
                const float2 ei = comp == 0 ? make_float2(xa.y, xb.y) : dup2(ya.y);
#pragma unroll
                for (int m = 0; m < H; ++m) {
                    const float2 kz = make_float2(kz_[Line::e0(j, m)], kz_[Line::e1(j, m)]);
                    const float2 k2 = fma2(kz, kz, kxy);
                    float2 f;
                    if (OP == OP_Z_ABS) {              // k^{y-2} / k^{y-1}, 0 at k = 0
                        const float2 rel = mul2(k2, dup2(g.inv_kmax2));
                        const float2 ex = mul2(dup2(g.abs_e[comp]), make_float2(log2f(rel.x), log2f(rel.y)));
                        f = mul2(make_float2(ex2_normal(ex.x), ex2_normal(ex.y)), dup2(g.abs_c[comp] * g.scale));
                        if (!(k2.x > 0.f)) f.x = 0.f;
                        if (!(k2.y > 0.f)) f.y = 0.f;
                    } else {
                        const float2 x2 = mul2(dup2(g.hk2), k2);
                        f = mul2(a.short_kappa ? sinc_short2(x2) : sinc_any2(x2), dup2(g.scale));
                    }
                    if (ZD) {
                        float2 zr, zi;
                        dz(m, zr, zi);
                        cmul2(re[m], im[m], zr, zi);
                    } else if (OP == OP_Z_DIV || OP == OP_Z_DIV_FWD || SUM) {
                        cmul2(re[m], im[m], er, ei);
                    }
                    re[m] = mul2(re[m], f);
                    im[m] = mul2(im[m], f);
                }
            };
            if ((OP == OP_Z_DIV || OP == OP_Z_DIV_FWD || SUM) && comp == 2) apply(std::true_type{});
            else apply(std::false_type{});
            if (GRAD) stash_put(taddr, re, im);
            if (SUM) {
                // (the stashed values beside the live ones: up to 60 bytes of spill loads a thread, 618 for 256-point lines)
                if (comp > 0) {
                    float2 sr[H], si[H];
                    stash_get(taddr, sr, si);
#pragma unroll
                    for (int m = 0; m < H; ++m) {
                        re[m] = add2(sr[m], re[m]);
                        im[m] = add2(si[m], im[m]);
                    }
                }
                if (comp < 2) {
                    stash_put(taddr, re, im);
                    next();
                    continue;
                }
            }
            if (GRAD) {
                // kappa is common to the three outputs, and the x and y shift operators do not
                // vary along z: outputs 0 and 1 are dx Q and dy Q with Q = IFT_z{kappa P}; output 2
                // is the inverse transform of kappa dz P, taken from the stash
                if (a.out[0] != nullptr || a.out[1] != nullptr) {         // uniform
                    Line::inv(re, im, buf, c, j, tw, sync);
                    Line::inv_end(re, im, j, [&](int ea, int eb, float2 va, float2 vb) {
                        const size_t o = off + (size_t)ea * es, step = (size_t)(eb - ea) * es;
                        if (a.out[0] != nullptr) Line::store(a.out[0] + o, step, cmul(va, xa), cmul(vb, xb), v0, v1);
                        if (a.out[1] != nullptr) Line::store(a.out[1] + o, step, cmul(va, ya), cmul(vb, ya), v0, v1);
                    });
                }
                if (a.out[2] == nullptr) {
                    next();
                    continue;
                }
                stash_get(taddr, re, im);
#pragma unroll
                for (int m = 0; m < H; ++m) {
                    float2 zr, zi;
                    dz(m, zr, zi);
                    cmul2(re[m], im[m], zr, zi);
                }
            }
            Line::inv(re, im, buf, c, j, tw, sync);
            next();
            float2* out = out_ptr(a, GRAD ? 2 : (SUM ? 0 : comp)) + off;
            Line::inv_end(re, im, j, [&](int ea, int eb, float2 va, float2 vb) {
                Line::store(out + (size_t)ea * es, (size_t)(eb - ea) * es, va, vb, v0, v1);
            });
        }
    }
    }
    if (__syncthreads_or(gave_up) && threadIdx.x < 4 * GR) {  // every group has finished or given up
        // A load is issued when the one NBUF before it has been released, and a group releases its loads
        // in order, up to stop[].  The loads of a group beyond that which are issued are among its next
        // three (the groups feed each other in pairs): one to a lane, so that the waits run side by side.
        const int gr = threadIdx.x / 4;
        const int n = stop[gr] / (PER * GR) * PER + stop[gr] % PER + threadIdx.x % 4;   // the group's n-th load
        const int q = (n / PER * GR + gr) * PER + n % PER;
        const int feeder = (q - NBUF) / PER % GR;
        if (stop[gr] >= 0 && q < Q && (q < NBUF || stop[feeder] < 0 || q - NBUF < stop[feeder]))
            mbar_wait_bounded(&bar[q % (2 * NBUF)], (q / (2 * NBUF)) & 1, a.flag);
    }
    if (STASH) {
        tc5_fence_before();
        __syncthreads();
        tc5_fence_after();
        if (threadIdx.x < 32) tc5_dealloc(tslot, 256);
    }
}

template <int LOGN, int OP>
inline cudaError_t launch_line(const YZK& a, cudaStream_t s) {
    using Ls = LShape<LOGN, (OP < 2)>;
    constexpr bool stash = OP == OP_Z_GRAD_FWD || OP == OP_Z_GRAD_BWD || OP == OP_Z_DIV_SUM;
    auto k = line_kernel<LOGN, OP>;
    static PerDevice ready;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    ready.get(dev, [&] {
        e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, Ls::SMEM);
        return e == cudaSuccess ? 1 : 0;
    });
    if (e != cudaSuccess) return e;
    const int nchunk = (a.g.nh + Ls::Sh::CX - 1) / Ls::Sh::CX;
    const int lines = OP < 2 ? a.g.nz : a.g.ny;
    const int units = nchunk * lines * (OP < 2 ? a.ncomp : (stash ? 1 : a.nloads));
    const int grid = std::min(a.g.num_sms, units);
    if (grid < 1) return cudaSuccess;
    return launch_after(k, grid, 512, Ls::SMEM, s, a);
}

}  // namespace kwgb
