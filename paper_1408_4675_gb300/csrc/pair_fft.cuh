// Two FFT lines at once in packed float32 arithmetic.
//
// Blackwell executes add, mul and fma on a pair of float32 values held in one
// 64-bit register as a single instruction (PTX add/mul/fma.rn.f32x2), with
// the rounding of the scalar instructions.  The strided passes are bound by
// instruction issue, so a thread that holds two lines keeps them as pairs:
//   re[m] = (real part of line a, real part of line b), im[m] likewise,
// and every butterfly, twiddle and operator product of both lines is one
// instruction instead of two.  The inverse transform is the forward one with
// the roles of re and im swapped (DFT+ x = swap(DFT- (swap x))), which costs
// nothing in this form, so only the forward butterflies exist.
#pragma once

#include "fft_core.cuh"

namespace kwgb {

__device__ __forceinline__ unsigned long long p2u(float2 a) { return reinterpret_cast<unsigned long long&>(a); }
__device__ __forceinline__ float2 u2p(unsigned long long a) { return reinterpret_cast<float2&>(a); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(p2u(a)), "l"(p2u(b)));
    return u2p(r);
}
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
    unsigned long long r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(p2u(a)), "l"(p2u(b)));
    return u2p(r);
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
    unsigned long long r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(p2u(a)), "l"(p2u(b)));
    return u2p(r);
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(p2u(a)), "l"(p2u(b)), "l"(p2u(c)));
    return u2p(r);
}
__device__ __forceinline__ float2 dup2(float s) { return make_float2(s, s); }
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }

// (re, im) *= (c + i s), packed: re' = re c - im s, im' = im c + re s.  Of each sum's two products one
// is rounded by itself, the other within the fma; better the smaller one, so constant factors nearer
// to 1 than to i take cmul2_flat.  (For table twiddles it makes no difference that can be measured, and the
// other order costs the 512-point gradient pass registers: 1.985 -> 2.047 ms at 512^3.)
__device__ __forceinline__ void cmul2(float2& re, float2& im, float2 c, float2 s) {
    const float2 r = fma2(im, neg2(s), mul2(re, c));
    im = fma2(re, s, mul2(im, c));
    re = r;
}
__device__ __forceinline__ void cmul2_flat(float2& re, float2& im, float2 c, float2 s) {
    const float2 r = fma2(re, c, mul2(im, neg2(s)));
    im = fma2(im, c, mul2(re, s));
    re = r;
}

// exp(-2 pi i m / 16) is nearer to +-i than to +-1
__host__ __device__ constexpr bool steep16(int m) { return (m & 7) > 2 && (m & 7) < 6; }

// (re, im) *= exp(-2 pi i m / 16) for a compile-time m in [0, 16), m != 8, 12.
__device__ __forceinline__ void rot2(float2& re, float2& im, int m) {
    if (m == 0) return;
    if (m == 4) {                                     // * -i
        const float2 r = im;
        im = neg2(re);
        re = r;
        return;
    }
    if (steep16(m)) cmul2(re, im, dup2(cos16(m)), dup2(-sin16(m)));
    else cmul2_flat(re, im, dup2(cos16(m)), dup2(-sin16(m)));
}

// Forward DFT of four values at a, b, c, d, in place (output k in the k-th).
__device__ __forceinline__ void dft4_pair(float2* re, float2* im, int a, int b, int c, int d) {
    const float2 s0 = add2(re[a], re[c]), t0 = add2(im[a], im[c]), s1 = sub2(re[a], re[c]), t1 = sub2(im[a], im[c]);
    const float2 s2 = add2(re[b], re[d]), t2 = add2(im[b], im[d]), s3 = sub2(re[b], re[d]), t3 = sub2(im[b], im[d]);
    re[a] = add2(s0, s2);
    im[a] = add2(t0, t2);
    re[b] = add2(s1, t3);
    im[b] = sub2(t1, s3);
    re[c] = sub2(s0, s2);
    im[c] = sub2(t0, t2);
    re[d] = sub2(s1, t3);
    im[d] = add2(t1, s3);
}

// Sixteen values as 4 x 4: 8 of them are rotated (and rounded) once, against 10 rotations in the
// radix-2 form; with those a line of 512 points was less accurate than three radix-8 passes
// (1.08e-7 relative error against 1.02e-7; now 1.05e-7, and 1.04e-7 with the order of cmul2_flat).
__device__ __forceinline__ void dft16_pair(float2* re, float2* im) {
#pragma unroll
    for (int n = 0; n < 4; ++n) {
        dft4_pair(re, im, n, n + 4, n + 8, n + 12);
#pragma unroll
        for (int k = 1; k < 4; ++k) rot2(re[n + 4 * k], im[n + 4 * k], n * k);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) dft4_pair(re, im, 4 * k, 4 * k + 1, 4 * k + 2, 4 * k + 3);   // output k + 4 q at 4 k + q
    float2 t[16], u[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        t[i] = re[4 * (i & 3) + (i >> 2)];
        u[i] = im[4 * (i & 3) + (i >> 2)];
    }
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        re[i] = t[i];
        im[i] = u[i];
    }
}

// In-register forward DFT of size R on two lines (dft_reg in pair form).
template <int R>
__device__ __forceinline__ void dft_pair(float2* re, float2* im) {
    static_assert(R == 1 || R == 2 || R == 4 || R == 8 || R == 16, "radix");
    if constexpr (R == 16) {
        dft16_pair(re, im);
        return;
    }
    constexpr int LR = ilog2c(R);
#pragma unroll
    for (int st = 0; st < LR; ++st) {
        const int span = R >> (st + 1);
#pragma unroll
        for (int g = 0; g < (1 << st); ++g) {
#pragma unroll
            for (int j = 0; j < (R >> (st + 1)); ++j) {
                const int a = g * 2 * span + j, b = a + span;
                const int m = j * (16 / (2 * span));
                const float2 ar = re[a], ai = im[a], br = re[b], bi = im[b];
                re[a] = add2(ar, br);
                im[a] = add2(ai, bi);
                if (m == 4) {                         // (x - y) * -i without a negation
                    re[b] = sub2(ai, bi);
                    im[b] = sub2(br, ar);
                } else {
                    re[b] = sub2(ar, br);
                    im[b] = sub2(ai, bi);
                    rot2(re[b], im[b], m);
                }
            }
        }
    }
    if (R > 2) {
        float2 t[R], u[R];
#pragma unroll
        for (int i = 0; i < R; ++i) {
            t[i] = re[bitrev(i, LR)];
            u[i] = im[bitrev(i, LR)];
        }
#pragma unroll
        for (int i = 0; i < R; ++i) {
            re[i] = t[i];
            im[i] = u[i];
        }
    }
}

}  // namespace kwgb
