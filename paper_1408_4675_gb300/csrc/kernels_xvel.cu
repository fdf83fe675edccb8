// x_vel: C2R of the three gradient spectra (Eq. 4a) -> velocity update with
// PML (Eq. 4b) and force sources -> R2C of the new u_xi (first stage of
// Eq. 4c).  Row layout and helpers: x_rows.cuh.
#include "x_rows.cuh"

namespace kwgb {

// One row per TL threads per launch slot (not persistent).
struct XVelK {
    GridC g;
    Medium md;
    XVelArgs a;
};

// FORCE: the launch has force sources (a separate instantiation, so that the
// common path carries no code for them).  ONE: a CTA takes one component of its
// rows (blockIdx mod 3) instead of all three one after another.
template <int LOGM, int MODE, bool FORCE, bool ONE>
__global__ void __launch_bounds__(XShape<LOGM>::XT, XShape<LOGM>::MINB) x_vel_kernel(const XVelK K) {
    using Sh = XShape<LOGM>;
    constexpr int E = Sh::E, TL = Sh::TL;
    extern __shared__ float2 smem[];
    const GridC& g = K.g;
    const int r = threadIdx.x / TL, j = threadIdx.x % TL;
    const int nrows = g.ny * g.nz;
    const int row = (ONE ? blockIdx.x / 3 : blockIdx.x) * Sh::RPB + r;
    const bool valid = row < nrows;
    const int rr = valid ? row : 0;
    const int y = rr % g.ny, z = rr / g.ny;
    typename Sh::Smem S = Sh::row_smem(smem, r);
    const size_t rb = (size_t)rr * g.nx;
    const float* rho0 = K.md.rho0;
    const float rho0s = K.md.rho0_s;

    float2 r0[E];                                     // rho0 of this row (x = 2n, 2n+1)
#pragma unroll
    for (int m = 0; m < E; ++m) r0[m] = rho0 ? ldg2(rho0 + rb + 2 * (j + TL * m)) : make_float2(rho0s, rho0s);
    after_previous();
    auto component = [&](int xi) {
        // issue this component's field loads before the row transform
        size_t nb;                                    // row base of the +1 neighbour along y / z
        if (xi == 1) nb = (size_t)(((y + 1) & (g.ny - 1)) + g.ny * z) * g.nx;
        else nb = (size_t)(y + g.ny * ((z + 1) & (g.nz - 1))) * g.nx;
        float* u = pick3f(K.a.u, xi);
        float2 uo[E], r1[E];
#pragma unroll
        for (int m = 0; m < E; ++m) {
            const int x = 2 * (j + TL * m);
            uo[m] = (MODE != XV_INIT && valid) ? ld2(u + rb + x) : make_float2(0.f, 0.f);
            if (!rho0) r1[m] = make_float2(rho0s, rho0s);
            else if (xi == 0) r1[m] = make_float2(__ldg(rho0 + rb + ((x + 2) & (g.nx - 1))), 0.f);
            else r1[m] = ldg2(rho0 + nb + x);
        }
        float2 v[E];
        row_c2r<LOGM>(spec_row<Sh::M>(pick3(K.a.G, xi), rr), g, S, j, valid, g.t.tw, v);
        const float fyz = xi == 1 ? __ldg(g.t.pml_sg[1] + y) : __ldg(g.t.pml_sg[2] + z);
#pragma unroll
        for (int m = 0; m < E; ++m) {
            const int x = 2 * (j + TL * m);
            // staggered-grid density: mean of the two neighbours along xi
            const float2 n1 = xi == 0 ? make_float2(r0[m].y, rho0 ? r1[m].x : rho0s) : r1[m];
            const float2 rs = make_float2(0.5f * (r0[m].x + n1.x), 0.5f * (r0[m].y + n1.y));
            const float2 f = xi == 0 ? ldg2(g.t.pml_sg[0] + x) : make_float2(fyz, fyz);
            const float2 gr = v[m];
            float2 un;
            if (MODE == XV_INIT) {
                // u^{-1/2} = +dt / (2 rho0_sg) d/dxi p0
                un = make_float2(__fdividef(0.5f * g.dt * gr.x, rs.x), __fdividef(0.5f * g.dt * gr.y, rs.y));
            } else {
                // Eq. 4b with the PML: u <- f (f u - dt grad p / rho0_sg)
                un = make_float2(f.x * (f.x * uo[m].x - __fdividef(g.dt * gr.x, rs.x)),
                                 f.y * (f.y * uo[m].y - __fdividef(g.dt * gr.y, rs.y)));
            }
            if (valid) {
                if (MODE == XV_TAIL) __stcs(spec_at<Sh::M>(spec_row<Sh::M>(reinterpret_cast<float2*>(pick3f(K.a.tail, xi)), rr), g, x >> 1), un);
                else st2(u + rb + x, un);
            }
            v[m] = un;
        }
        const SourceC& fs = xi == 0 ? K.a.f[0] : (xi == 1 ? K.a.f[1] : K.a.f[2]);
        if (FORCE && MODE != XV_INIT && fs.row_ptr) {   // force sources along xi (uniform over the CTA)
            // u_xi += dt F / rho0_sg at the row's source points, after Eq. 4b; the
            // point's value (already stored above) is stored again by its thread
            const int p0 = valid ? __ldg(fs.row_ptr + rr) : 0, p1 = valid ? __ldg(fs.row_ptr + rr + 1) : 0;
            S.sync();
            if (p1 > p0) {
#pragma unroll
                for (int m = 0; m < E; ++m) {
                    const int x = 2 * (j + TL * m);
                    S.f(x) = v[m].x;
                    S.f(x + 1) = v[m].y;
                }
            }
            S.sync();
            if (p1 > p0) {
                const int64_t n = *K.a.step;
                for_row_sources<TL>(
                    fs, p0, p1, j, n,
                    [&](int x) {                      // rho0 at the staggered point x + 1/2 along xi
                        if (!rho0) return rho0s;
                        const size_t other = xi == 0 ? rb + ((x + 1) & (g.nx - 1)) : nb + x;
                        return 0.5f * (__ldg(rho0 + rb + x) + __ldg(rho0 + other));
                    },
                    [&](int x, float acc, bool, float rsx) {
                        const float un = S.f(x) + __fdividef(acc, rsx);
                        S.f(x) = un;
                        if (MODE == XV_TAIL)
                            reinterpret_cast<float*>(spec_at<Sh::M>(spec_row<Sh::M>(reinterpret_cast<float2*>(pick3f(K.a.tail, xi)), rr), g, x >> 1))[x & 1] = un;
                        else u[rb + x] = un;
                    });
            }
            S.sync();
            if (p1 > p0) {
#pragma unroll
                for (int m = 0; m < E; ++m) {
                    const int x = 2 * (j + TL * m);
                    v[m] = make_float2(S.f(x), S.f(x + 1));
                }
            }
        }
        if (MODE == XV_STEP) row_r2c<LOGM>(v, S, j, valid, g.t.tw, spec_row<Sh::M>(pick3w(K.a.U, xi), rr), g);
    };
    if (ONE) component(blockIdx.x % 3);
    else {
#pragma unroll
        for (int xi = 0; xi < 3; ++xi) component(xi);
    }
}

// All three components in one CTA read rho0 once (512^3: 1.39 ms against 1.53 ms
// with a component per CTA).  Where those CTAs would not even fill the SMs once,
// the components' latencies in a row are the kernel's time, and one
// component per CTA is faster (32^3 10.2 -> 8.2 us, 32 x 256 x 128 21.4 -> 19.9 us;
// 128^3, 1.7 times the slots: 28.9 and 27.9 us).
template <int L, bool FORCE>
static cudaError_t launch_step_vel(const GridC& g, const XVelK& K, cudaStream_t s) {
    using Sh = XShape<L>;
    const int ctas = (g.ny * g.nz + Sh::RPB - 1) / Sh::RPB;
    if (ctas <= Sh::MINB * g.num_sms) return launch_rows<L>(x_vel_kernel<L, XV_STEP, FORCE, true>, Sh::SMEM, g, K, s, 3);
    return launch_rows<L>(x_vel_kernel<L, XV_STEP, FORCE, false>, Sh::SMEM, g, K, s);
}

cudaError_t launch_x_vel(const GridC& g, const Medium& m, int mode, const XVelArgs& a,
                         cudaStream_t s) {
    XVelK K{g, m, a};
    const bool force = a.f[0].row_ptr || a.f[1].row_ptr || a.f[2].row_ptr;
    switch (g.lognx - 1) {
#define CASE(L)                                                                                   \
    case L:                                                                                       \
        if (mode == XV_STEP) return force ? launch_step_vel<L, true>(g, K, s) : launch_step_vel<L, false>(g, K, s); \
        if (mode == XV_TAIL && force) return launch_rows<L>(x_vel_kernel<L, XV_TAIL, true, false>, XShape<L>::SMEM, g, K, s); \
        if (mode == XV_TAIL) return launch_rows<L>(x_vel_kernel<L, XV_TAIL, false, false>, XShape<L>::SMEM, g, K, s); \
        return launch_rows<L>(x_vel_kernel<L, XV_INIT, false, false>, XShape<L>::SMEM, g, K, s);
        KWGB_LOGM_CASES(CASE)
#undef CASE
    }
    return cudaErrorInvalidValue;
}

}  // namespace kwgb
