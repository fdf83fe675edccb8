// Shared parts of the contiguous-axis (x) passes (kernels_xvel.cu,
// kernels_x.cu): complex-to-real and real-to-complex transforms
// of whole rows, fused with the pointwise work of the time step so that the
// real-space fields only ever exist in registers:
//
//   x_vel   C2R of the three gradient spectra (Eq. 4a) -> velocity update with
//           PML (Eq. 4b) -> R2C of the new u_xi (first stage of Eq. 4c)
//   x_dens  C2R of the three divergence spectra (Eq. 4c) -> split density
//           update with PML and nonlinear denominator (Eq. 4d) -> additive
//           mass source -> rho = sum rho_xi and rho0 sum d -> R2C of both
//           (first stage of Eq. 8); for a lossless medium the EOS (Eq. 6),
//           the sensors and the R2C of p are done here as well
//   x_eos   C2R of the two absorption spectra (Eq. 8) -> EOS (Eq. 6) ->
//           sensors -> R2C of p^{n+1} (first stage of the next Eq. 4a)
//
// A row of nx reals is treated as M = nx/2 complex values z[n] = x[2n] +
// i x[2n+1]; an M-point FFT plus one post-processing step pairing bins k and
// M-k gives the nx/2+1 bins of the real transform (and the reverse for C2R).
// TL = M/E threads own a row; thread j holds z[j + TL*m], i.e. the float2 at
// x = 2(j + TL*m), so every global access of a row is coalesced.  A "team"
// is the smallest set of whole warps that holds whole rows: one warp with
// 32/TL rows (TL <= 32), or the TL/32 warps of one row (1024-point rows:
// E = 8, TL = 64, two warps, so that the kernels keep 16 warps per SM
// instead of spilling 16 values per thread in half as many).  All synchronisation
// is within a team (a warp barrier, or a named barrier per team), so the
// teams of a CTA stream their rows independently.
#pragma once

#include "fft_core.cuh"
#include "kwgb_internal.h"
#include "launch.cuh"

namespace kwgb {


// Element k of a row's spectrum (or real row kept in a spectrum buffer); row: the
// row's element 0 (spec_row), M: half the row length.  (The block width is a
// constant of the row length, so that k = j + TL m costs one base and a multiple.)
template <int M, class T>
__device__ __forceinline__ T* spec_at(T* row, const GridC& g, int k) {
    constexpr int LB = spec_block_log2(2 * M);
    return row + (((size_t)g.ny * g.nz) << LB) * (k >> LB) + (k & ((1 << LB) - 1));
}
template <int M, class T>
__device__ __forceinline__ T* spec_row(T* spec, int row) { return spec + ((size_t)row << spec_block_log2(2 * M)); }

// Work row of a team in shared memory, and the team's barrier.  TEAMS: teams per CTA.
// The barrier ids are literals: with an id in a register the compiler reserves all 16 barriers
// for a CTA, and the SM's barriers then limit how many of the small CTAs of the plain
// x transforms it holds (gradient of 256 x 512 x 1024, three literal barriers instead of 16:
// 2.22 -> 1.95 ms, eta of 64 x 512 x 1024 258 -> 226 us, step of 1024^3 65.3 -> 64.8 ms).
template <int TEAM, int TEAMS>
struct RowSmem {
    float2* base;
    int team;                                        // this team (TEAM > 32)
    static constexpr bool PINGPONG = false;
    __device__ __forceinline__ float2& at(int e) { return base[e + (e >> 4)]; }
    __device__ __forceinline__ float& f(int x) { return reinterpret_cast<float*>(base)[x]; }
    __device__ __forceinline__ void sync() {
        static_assert(TEAM <= 32 || TEAMS == 2, "one barrier per team");
        if constexpr (TEAM <= 32) __syncwarp();
        else if (team == 0) asm volatile("bar.sync 1, %0;" ::"n"(TEAM) : "memory");
        else asm volatile("bar.sync 2, %0;" ::"n"(TEAM) : "memory");
    }
};

template <int LOGM>
struct XShape {
    static constexpr int M = 1 << LOGM;
    static constexpr int E = M >= 8 ? 8 : M;
    static constexpr int TL = M / E;
    static constexpr int TEAM = TL > 32 ? TL : 32;   // threads of a team
    // threads of a CTA.  The warps of a CTA work on rows of their own, but its slot
    // is free only when the last one has finished, and short rows come with small grids,
    // where CTAs of 256 threads (up to 128 rows) would leave most SMs without one.  Measured:
    // x_eos 512^3 876 -> 800 us and 1024^3 7.25 -> 6.86 ms with 128 threads instead of 256 (64: 804 us; x_vel,
    // which reads rho0 of the rows above, 1.33 -> 1.34 ms), step 256^3 1017 -> 997 us with 64 (128: 1008),
    // x_vel 32^3 17.8 -> 10.2 us with 64 instead of 256.
    static constexpr int XT = LOGM <= 7 ? 64 : 128;
    static constexpr int RPT = TEAM / TL;            // rows per team
    static constexpr int TPB = XT / TEAM;      // teams per CTA
    static_assert(TPB >= 1, "a CTA holds whole teams");
    static constexpr int MINB = 512 / XT;            // resident CTAs per SM the fused kernels are compiled for
    static constexpr bool SHFL = TL <= 32;           // pairing steps by shuffles (mirrored)
    static constexpr int RPB = XT / TL;        // rows per CTA
    static constexpr int PITCH = M + M / 16 + 2;     // complex slots per row (padded, + Nyquist)
    static constexpr int SMEM = RPB * PITCH * (int)sizeof(float2);
    using Smem = RowSmem<TEAM, TPB>;
    // the work row of row slot r (threads r*TL .. r*TL + TL - 1) of a CTA
    __device__ __forceinline__ static Smem row_smem(float2* smem, int r) {
        return Smem{smem + r * PITCH, (r * TL) / TEAM};
    }
};

// exp(DIR 2 pi i k / (2M)) for k = j + TL*m, by FORM:
//   TW_TABLE  the table entry of k
//   TW_HALF   the entries of the first half of the m, the others those times DIR i (TL / M = 1 / E): as
//             accurate, half the loads
//   TW_ONE    one load per thread (w0 = the value at k = j) times the compile-time root
//             exp(DIR i pi m / E); the root's rounding and the product's come on top
enum { TW_TABLE, TW_HALF, TW_ONE };
template <int FORM, int DIR, int M, int E>
__device__ __forceinline__ float2 row_tw(const float2* __restrict__ tw, float2 w0, int k, int m) {
    static_assert(E <= 8 && 8 % E == 0, "roots of 16");
    if constexpr (FORM == TW_ONE) return rot16<DIR>(w0, m * (8 / E));
    if constexpr (FORM == TW_HALF) {
        if (m < E / 2) return row_twiddle<DIR, M>(tw, k);
        const float2 w = row_twiddle<DIR, M>(tw, k - M / 2);
        return DIR > 0 ? make_float2(-w.y, w.x) : make_float2(w.y, -w.x);
    }
    return row_twiddle<DIR, M>(tw, k);
}
template <int FORM, int DIR, int M>
__device__ __forceinline__ float2 row_tw0(const float2* __restrict__ tw, int j) {
    if constexpr (FORM == TW_ONE) return row_twiddle<DIR, M>(tw, j);
    else return make_float2(0.f, 0.f);
}
// Rows of 1024 reals: one load; 512: half the loads (step of 512^3 7.36 ms, with the table 7.46, with one
// load 7.37); shorter rows: the table (256^3 0.963 ms, half the loads 0.976, one load 0.960).  One load
// below 1024 reals cost accuracy: error of gradients of 64 x 64 x 512 against float64 4.08e-7 -> 4.11e-7, of a
// step's p_max at 256^3 3.09e-7 -> 3.20e-7.
template <int M>
__host__ __device__ constexpr int tw_form() { return M >= 512 ? TW_ONE : (M >= 256 ? TW_HALF : TW_TABLE); }

// Unnormalised C2R of one row: spec[0..M] (Hermitian half spectrum) ->
// z[m] = (x[2n], x[2n+1]) with n = j + TL*m and
// x[i] = sum_{k<nx} X[k] exp(+2 pi i k i / nx).
template <int LOGM>
__device__ __forceinline__ void row_c2r_lds(const float2* __restrict__ spec, const GridC& g, typename XShape<LOGM>::Smem& S, int j,
                                        bool valid, const float2* __restrict__ tw,
                                        float2 (&z)[XShape<LOGM>::E]) {
    using Sh = XShape<LOGM>;
    constexpr int M = Sh::M, E = Sh::E, TL = Sh::TL;
    // all E + 1 loads of the row are issued before the first one is used
    float2 t[E];
    float2 nyq = make_float2(0.f, 0.f);
#pragma unroll
    for (int m = 0; m < E; ++m) t[m] = valid ? __ldcs(spec_at<M>(spec, g, j + TL * m)) : make_float2(0.f, 0.f);
    if (valid && j == 0) nyq = __ldcs(spec_at<M>(spec, g, M));
    S.sync();                                      // smem row free
#pragma unroll
    for (int m = 0; m < E; ++m) S.at(j + TL * m) = t[m];
    if (j == 0) S.at(M) = nyq;
    S.sync();
    const float2 w0 = row_tw0<TW_ONE, +1, M>(tw, j);
#pragma unroll
    for (int m = 0; m < E; ++m) {
        const int k = j + TL * m;
        const float2 xk = S.at(k), xm = cconj(S.at(M - k));
        const float2 a = cadd(xk, xm);
        const float2 b = cmul(csub(xk, xm), row_tw<TW_ONE, +1, M, E>(tw, w0, k, m));   // exp(+2 pi i k / nx)
        z[m] = make_float2(a.x - b.y, a.y + b.x);                                // a + i b
    }
    line_fft<LOGM, E, +1>(z, j, S, tw);
}

// The partner of element k in the pairing steps is element M - k: for k = j + TL m
// that is register E - 1 - m of lane TL - j (lane 0: its own register E - m), so a
// row within one warp gets it by a shuffle, which moves half the bytes of a round
// trip through shared memory (x_vel is bound by that data path, 80 % busy: 512^3
// 1.38 -> 1.33 ms, 128^3 26.4 -> 23.5 us).
template <int TL, int E>
__device__ __forceinline__ float2 mirrored(const float2 (&t)[E], float2 first, int j, int m) {
    float2 o;
    o.x = __shfl_sync(0xffffffffu, t[E - 1 - m].x, (TL - j) & (TL - 1), TL);
    o.y = __shfl_sync(0xffffffffu, t[E - 1 - m].y, (TL - j) & (TL - 1), TL);
    if (j == 0) o = m == 0 ? first : t[E - m > E - 1 ? 0 : E - m];
    return o;
}
template <int LOGM>
__device__ __forceinline__ void row_c2r_shfl(const float2* __restrict__ spec, const GridC& g, typename XShape<LOGM>::Smem& S, int j,
                                             bool valid, const float2* __restrict__ tw, float2 (&z)[XShape<LOGM>::E]) {
    using Sh = XShape<LOGM>;
    constexpr int M = Sh::M, E = Sh::E, TL = Sh::TL;
    float2 t[E];
    float2 nyq = make_float2(0.f, 0.f);
#pragma unroll
    for (int m = 0; m < E; ++m) t[m] = valid ? __ldcs(spec_at<M>(spec, g, j + TL * m)) : make_float2(0.f, 0.f);
    if (valid && j == 0) nyq = __ldcs(spec_at<M>(spec, g, M));
#pragma unroll
    for (int m = 0; m < E; ++m) {
        const int k = j + TL * m;
        const float2 xm = cconj(mirrored<TL, E>(t, nyq, j, m));
        const float2 a = cadd(t[m], xm);
        const float2 b = cmul(csub(t[m], xm), row_twiddle<+1, M>(tw, k));   // exp(+2 pi i k / nx)
        z[m] = make_float2(a.x - b.y, a.y + b.x);                                  // a + i b
    }
    line_fft<LOGM, E, +1>(z, j, S, tw);
}
template <int LOGM, int FORM>
__device__ __forceinline__ void row_r2c_shfl(float2 (&z)[XShape<LOGM>::E], typename XShape<LOGM>::Smem& S, int j,
                                             bool valid, const float2* __restrict__ tw, float2* __restrict__ spec, const GridC& g) {
    using Sh = XShape<LOGM>;
    constexpr int M = Sh::M, E = Sh::E, TL = Sh::TL;
    line_fft<LOGM, E, -1>(z, j, S, tw);
    const float2 w0 = row_tw0<FORM, -1, M>(tw, j);
#pragma unroll
    for (int m = 0; m < E; ++m) {
        const int k = j + TL * m;
        const float2 zm = cconj(mirrored<TL, E>(z, z[0], j, m));
        const float2 s = cadd(z[m], zm), d = csub(z[m], zm);
        const float2 xe = make_float2(0.5f * s.x, 0.5f * s.y);
        const float2 xo = make_float2(0.5f * d.y, -0.5f * d.x);              // d / (2i)
        const float2 x = cadd(xe, cmul(xo, row_tw<FORM, -1, M, E>(tw, w0, k, m)));   // exp(-2 pi i k / nx)
        if (valid) {
            __stcs(spec_at<M>(spec, g, k), x);
            if (k == 0) __stcs(spec_at<M>(spec, g, M), csub(xe, xo));
        }
    }
}

// ---- asynchronous row staging (per-warp cp.async double buffer) ----------
// A warp's rows of one spectrum are copied into shared memory one item ahead
// of their use, so the global-memory latency of the row load overlaps the
// transform of the previous item.  Rows are copied as M + 2 complex values
// (a multiple of 16 bytes; the extra value lies in the row padding).
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
                 "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait1() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait0() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

template <int LOGM>
struct XStage {
    static constexpr int M = 1 << LOGM;
    static constexpr int SROW = M + 2;                   // staged complex values per row
    static constexpr int RPT = XShape<LOGM>::RPT;        // rows per team
    static constexpr int TEAM = XShape<LOGM>::TEAM;
    static constexpr int TSTAGE = 2 * RPT * SROW;        // complex per team (two stages)
};

// Issue the copies of rows first_row .. first_row + RPT - 1 of `spec` into
// stage buffer `dst` (RPT * SROW complex).  All threads of the team take part.
template <int LOGM>
__device__ __forceinline__ void stage_rows(float2* dst, const float2* __restrict__ spec, int first_row,
                                           int nrows, const GridC& g, int lane) {
    using St = XStage<LOGM>;
    constexpr int CH = St::SROW / 2;                     // 16-byte chunks per row
#pragma unroll
    for (int t = 0; t < (St::RPT * CH + St::TEAM - 1) / St::TEAM; ++t) {
        const int c = lane + St::TEAM * t;
        if (c < St::RPT * CH) {
            const int r = c / CH, q = c % CH;
            if (first_row + r < nrows)
                cp_async16(dst + r * St::SROW + 2 * q, spec_at<St::M>(spec_row<St::M>(spec, first_row + r), g, 2 * q));
        }
    }
}

// C2R of one row whose half spectrum X[0..M] is already in shared memory
// (srow, unpadded): same result as row_c2r.
template <int LOGM>
__device__ __forceinline__ void row_c2r_staged(const float2* srow, typename XShape<LOGM>::Smem& S, int j,
                                               const float2* __restrict__ tw,
                                               float2 (&z)[XShape<LOGM>::E]) {
    using Sh = XShape<LOGM>;
    constexpr int M = Sh::M, E = Sh::E, TL = Sh::TL;
    const float2 w0 = row_tw0<tw_form<M>(), +1, M>(tw, j);
#pragma unroll
    for (int m = 0; m < E; ++m) {
        const int k = j + TL * m;
        const float2 xk = srow[k], xm = cconj(srow[M - k]);
        const float2 a = cadd(xk, xm);
        const float2 b = cmul(csub(xk, xm), row_tw<tw_form<M>(), +1, M, E>(tw, w0, k, m));   // exp(+2 pi i k / nx)
        z[m] = make_float2(a.x - b.y, a.y + b.x);                                // a + i b
    }
    S.sync();                                        // previous users of the work row are done
    line_fft<LOGM, E, +1>(z, j, S, tw);
}

template <int LOGM, int FORM>
__device__ __forceinline__ void row_r2c_smem(float2 (&z)[XShape<LOGM>::E], typename XShape<LOGM>::Smem& S, int j,
                                        bool valid, const float2* __restrict__ tw,
                                        float2* __restrict__ spec, const GridC& g) {
    using Sh = XShape<LOGM>;
    constexpr int M = Sh::M, E = Sh::E, TL = Sh::TL;
    line_fft<LOGM, E, -1>(z, j, S, tw);
    S.sync();
#pragma unroll
    for (int m = 0; m < E; ++m) S.at(j + TL * m) = z[m];
    S.sync();
    if (valid) {
        const float2 w0 = row_tw0<FORM, -1, M>(tw, j);
#pragma unroll
        for (int m = 0; m < E; ++m) {
            const int k = j + TL * m;
            const float2 zk = z[m], zm = cconj(S.at((M - k) & (M - 1)));
            const float2 s = cadd(zk, zm), d = csub(zk, zm);
            const float2 xe = make_float2(0.5f * s.x, 0.5f * s.y);
            const float2 xo = make_float2(0.5f * d.y, -0.5f * d.x);              // d / (2i)
            const float2 x = cadd(xe, cmul(xo, row_tw<FORM, -1, M, E>(tw, w0, k, m)));   // exp(-2 pi i k / nx)
            __stcs(spec_at<M>(spec, g, k), x);
            if (k == 0) __stcs(spec_at<M>(spec, g, M), csub(xe, xo));
        }
    }
}

// Unnormalised R2C of one row: z[m] = (x[2n], x[2n+1]) -> spec[0..M].
template <int LOGM, int FORM = tw_form<(1 << LOGM)>()>
__device__ __forceinline__ void row_r2c(float2 (&z)[XShape<LOGM>::E], typename XShape<LOGM>::Smem& S, int j,
                                        bool valid, const float2* __restrict__ tw,
                                        float2* __restrict__ spec, const GridC& g) {
    if constexpr (XShape<LOGM>::SHFL) row_r2c_shfl<LOGM, FORM>(z, S, j, valid, tw, spec, g);
    else row_r2c_smem<LOGM, FORM>(z, S, j, valid, tw, spec, g);
}

template <int LOGM>
__device__ __forceinline__ void row_c2r(const float2* __restrict__ spec, const GridC& g, typename XShape<LOGM>::Smem& S, int j,
                                        bool valid, const float2* __restrict__ tw, float2 (&z)[XShape<LOGM>::E]) {
    if constexpr (XShape<LOGM>::SHFL) row_c2r_shfl<LOGM>(spec, g, S, j, valid, tw, z);
    else row_c2r_lds<LOGM>(spec, g, S, j, valid, tw, z);
}

__device__ __forceinline__ float2 ld2(const float* p) { return __ldcs(reinterpret_cast<const float2*>(p)); }
__device__ __forceinline__ float2 ldg2(const float* p) { return __ldg(reinterpret_cast<const float2*>(p)); }
__device__ __forceinline__ void st2(float* p, float2 v) { __stcs(reinterpret_cast<float2*>(p), v); }

__device__ __forceinline__ float2 med2(const float* f, float s, size_t i) {
    return f ? ldg2(f + i) : make_float2(s, s);
}

// Sensors, non-finite watch and the R2C of p (shared by x_eos and the fused
// lossless x_dens).  p[m] holds p at x = 2n, 2n+1.
template <int LOGM>
__device__ __forceinline__ void finish_pressure(float2 (&p)[XShape<LOGM>::E], const GridC& g,
                                                const SensorC& sens, const StepC& st,
                                                typename XShape<LOGM>::Smem& S, int j, bool valid, int row,
                                                float2* __restrict__ P) {
    using Sh = XShape<LOGM>;
    constexpr int E = Sh::E, TL = Sh::TL;
    const size_t rbase = (size_t)row * g.nx;
    if (valid) {
        bool bad = false;
#pragma unroll
        for (int m = 0; m < E; ++m) bad |= !(isfinite(p[m].x) && isfinite(p[m].y));
        if (bad) atomicOr(st.flag, 1);
        for (int k = 0; k < sens.nfull; ++k) {
            float* pm = sens.full_max[k] + rbase;
            double* p2 = sens.full_p2[k] + rbase;
            float* pn = sens.full_min[k] ? sens.full_min[k] + rbase : nullptr;
            // the row's loads before its stores: the compiler cannot tell that they do not overlap,
            // and one after another they were eight memory latencies
            float2 o[E];
            double2 q[E];
#pragma unroll
            for (int m = 0; m < E; ++m) {
                o[m] = *reinterpret_cast<float2*>(pm + 2 * (j + TL * m));
                q[m] = *reinterpret_cast<double2*>(p2 + 2 * (j + TL * m));
            }
#pragma unroll
            for (int m = 0; m < E; ++m) {
                const int x = 2 * (j + TL * m);
                *reinterpret_cast<float2*>(pm + x) = make_float2(fmaxf(o[m].x, p[m].x), fmaxf(o[m].y, p[m].y));
                q[m].x += (double)p[m].x * (double)p[m].x;
                q[m].y += (double)p[m].y * (double)p[m].y;
                *reinterpret_cast<double2*>(p2 + x) = q[m];
            }
            if (pn) {
#pragma unroll
                for (int m = 0; m < E; ++m) o[m] = *reinterpret_cast<float2*>(pn + 2 * (j + TL * m));
#pragma unroll
                for (int m = 0; m < E; ++m)
                    *reinterpret_cast<float2*>(pn + 2 * (j + TL * m)) = make_float2(fminf(o[m].x, p[m].x), fminf(o[m].y, p[m].y));
            }
        }
    }
    if (sens.row_ptr) {                               // uniform over the launch
        S.sync();
#pragma unroll
        for (int m = 0; m < E; ++m) {
            const int x = 2 * (j + TL * m);
            S.f(x) = p[m].x;
            S.f(x + 1) = p[m].y;
        }
        S.sync();
        if (valid) {
            const int e0 = __ldg(sens.row_ptr + row), e1 = __ldg(sens.row_ptr + row + 1);
            // U entries at a time: a row of a sensor plane has an entry at every x (slots differ, so
            // the order of the updates does not matter)
            constexpr int U = TL <= 8 ? 8 : 4;
            for (int b = e0 + j; b < e1; b += U * TL) {
                int slot[U], x[U];
                float pm[U];
                double p2[U];
#pragma unroll
                for (int i = 0; i < U; ++i) {
                    const bool in = b + i * TL < e1;
                    slot[i] = in ? __ldg(sens.e_slot + b + i * TL) : -1;
                    x[i] = in ? __ldg(sens.e_x + b + i * TL) : 0;
                }
#pragma unroll
                for (int i = 0; i < U; ++i) {
                    pm[i] = slot[i] >= 0 ? sens.p_max[slot[i]] : 0.f;
                    p2[i] = slot[i] >= 0 ? sens.p2[slot[i]] : 0.0;
                }
#pragma unroll
                for (int i = 0; i < U; ++i) {
                    if (slot[i] < 0) continue;
                    const float v = S.f(x[i]);
                    sens.p_max[slot[i]] = fmaxf(pm[i], v);
                    sens.p2[slot[i]] = p2[i] + (double)v * (double)v;
                    sens.p_sens[slot[i]] = v;
                }
            }
        }
    }
    row_r2c<LOGM>(p, S, j, valid, g.t.tw, spec_row<Sh::M>(P, row), g);
}

// The source points of one row in step n, shared out over the row's TL threads:
// f(x, sum, held, pre(x)) for each point, with the sum of its contributions
// that still have a sample (held: there is one).  The loads of U points are
// issued together: a row of a source plane has hundreds of them, and one after
// another (five dependent loads each) they took longer than the row itself
// (x_dens of a 128^3 step with a plane source 55 -> 45 us, of a 256^3 step 227 -> 185 us).
template <int TL, class Pre, class F>
__device__ __forceinline__ void for_row_sources(const SourceC& s, int e0, int e1, int j, int64_t n, Pre&& pre, F&& f) {
    constexpr int U = TL <= 8 ? 8 : 4;
    for (int b = e0 + j; b < e1; b += U * TL) {
        SrcEntry c[U];
        int before[U], after[U];
        float v[U], w[U];
#pragma unroll
        for (int i = 0; i < U; ++i) {
            const int e = b + i * TL;
            const int4 q = e < e1 ? __ldg(reinterpret_cast<const int4*>(s.ent + e)) : make_int4(-1, 0, 0, 0);
            c[i].x = q.x;
            c[i].nt = q.y;
            c[i].off = (int64_t)(((uint64_t)(uint32_t)q.w << 32) | (uint32_t)q.z);
            before[i] = e < e1 && e > e0 ? __ldg(&s.ent[e - 1].x) : -1;
            after[i] = e + 1 < e1 ? __ldg(&s.ent[e + 1].x) : -1;
        }
#pragma unroll
        for (int i = 0; i < U; ++i) {
            v[i] = n < c[i].nt ? __ldg(s.signal + c[i].off + n) * s.scale : 0.f;
            w[i] = c[i].x >= 0 ? pre(c[i].x) : 0.f;
        }
#pragma unroll
        for (int i = 0; i < U; ++i) {
            if (c[i].x < 0 || before[i] == c[i].x) continue;        // no entry, or not the point's first
            float acc = v[i];
            bool held = n < c[i].nt;
            if (after[i] == c[i].x) {
                for (int e = b + i * TL + 1; e < e1 && __ldg(&s.ent[e].x) == c[i].x; ++e)
                    if (n < __ldg(&s.ent[e].nt)) {
                        acc += __ldg(s.signal + __ldg(&s.ent[e].off) + n) * s.scale;
                        held = true;
                    }
            }
            f(c[i].x, acc, held, w[i]);
        }
    }
}

// Dirichlet pressure sources of one row in step n: afterwards S.f(x) holds the
// summed sample of every point x of the row that is held in this step, and
// NaN at every other x.  All threads of the row's team call it (it contains
// the team barriers); the result says whether the row has source points
// (the same for the threads of one row).
template <int LOGM>
__device__ __forceinline__ bool dirichlet_row(const SourceC& ds, const GridC& g, typename XShape<LOGM>::Smem& S,
                                              int j, bool valid, int row, int64_t n) {
    constexpr int TL = XShape<LOGM>::TL;
    const int p0 = valid ? __ldg(ds.row_ptr + row) : 0, p1 = valid ? __ldg(ds.row_ptr + row + 1) : 0;
    S.sync();
    if (p1 > p0) {
        for (int x = j; x < g.nx; x += TL) S.f(x) = __int_as_float(0x7fc00000);    // quiet NaN: not held
    }
    S.sync();
    for_row_sources<TL>(ds, p0, p1, j, n, [](int) { return 0.f; }, [&](int x, float acc, bool held, float) {
        if (held) S.f(x) = acc;
    });
    S.sync();
    return p1 > p0;
}

// p[i] for a run-time i without copying the parameter array to local memory
__device__ __forceinline__ const float2* pick3(const float2* const (&p)[3], int i) {
    return i == 0 ? p[0] : (i == 1 ? p[1] : p[2]);
}
__device__ __forceinline__ float* pick3f(float* const (&p)[3], int i) {
    return i == 0 ? p[0] : (i == 1 ? p[1] : p[2]);
}
__device__ __forceinline__ const float* pick3c(const float* const (&p)[3], int i) {
    return i == 0 ? p[0] : (i == 1 ? p[1] : p[2]);
}
__device__ __forceinline__ float2* pick3w(float2* const (&p)[3], int i) {
    return i == 0 ? p[0] : (i == 1 ? p[1] : p[2]);
}

// ---------------------------------------------------------------- launchers
// per_row: CTAs per group of rows (x_vel: one per component)
template <int LOGM, class Kern, class Args>
static cudaError_t launch_rows(Kern k, int smem_bytes, const GridC& g, const Args& args, cudaStream_t s, int per_row = 1) {
    using Sh = XShape<LOGM>;
    if (smem_bytes > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes);
        if (e != cudaSuccess) return e;
    }
    const int nrows = g.ny * g.nz;
    return launch_after(k, (nrows + Sh::RPB - 1) / Sh::RPB * per_row, Sh::XT, smem_bytes, s, args);
}

// Persistent launch of a pipelined row kernel: one CTA per resident slot.
template <int LOGM, class Kern, class Args>
static cudaError_t launch_persistent(Kern k, const GridC& g, const Args& args, cudaStream_t s) {
    using Sh = XShape<LOGM>;
    using St = XStage<LOGM>;
    const int smem_bytes = (Sh::RPB * Sh::PITCH + Sh::TPB * St::TSTAGE) * (int)sizeof(float2);
    int per_sm = 0;
    if (smem_bytes > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes);
        if (e != cudaSuccess) return e;
    }
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, Sh::XT, smem_bytes);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) per_sm = 1;
    const int ngroups = (g.ny * g.nz + Sh::RPT - 1) / Sh::RPT;
    int blocks = (ngroups + Sh::TPB - 1) / Sh::TPB;
    if (blocks > per_sm * g.num_sms) blocks = per_sm * g.num_sms;
    return launch_after(k, blocks, Sh::XT, smem_bytes, s, args);
}

#define KWGB_LOGM_CASES(X) X(2) X(3) X(4) X(5) X(6) X(7) X(8) X(9)

}  // namespace kwgb
