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

// (re, im) *= (c + i s), packed: re' = re c - im s, im' = im c + re s.
__device__ __forceinline__ void cmul2(float2& re, float2& im, float2 c, float2 s) {
    const float2 r = fma2(im, neg2(s), mul2(re, c));
    im = fma2(re, s, mul2(im, c));
    re = r;
}

// (re, im) *= exp(-2 pi i m / 16) for a compile-time m in [0, 8).
__device__ __forceinline__ void rot2(float2& re, float2& im, int m) {
    if (m == 0) return;
    if (m == 4) {                                     // * -i
        const float2 r = im;
        im = neg2(re);
        re = r;
        return;
    }
    cmul2(re, im, dup2(cos16(m)), dup2(-sin16(m)));
}

// In-register forward DFT of size R on two lines (dft_reg in pair form).
template <int R>
__device__ __forceinline__ void dft_pair(float2* re, float2* im) {
    static_assert(R == 1 || R == 2 || R == 4 || R == 8 || R == 16, "radix");
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
