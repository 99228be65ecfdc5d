// The FP64 iterations on 64-bit fixed point (lgf_fx.cuh): start and end of a
// loop, the update and the Delta stencil.  Arrays of a loop:
//   UX   [mu=4][6][V]  rows 0,1 of every link, x 2^61 (whatever form the context
//                      stores its FP64 links in)
//   GX   [6][V]        rows 0,1 of G, x 2^61 (null: not tracked)
//   gX   [9][V]        g, x 2^61
//   AHX  [mu=4][4][V]  packed anti-Hermitian parts of the links, x 2^57; the
//                      fourth entry holds 2 Im w00 - Im w11 - Im w22 and 2 Im w11
//                      - Im w00 - Im w22 (3/2 of the packed traceless diagonal:
//                      the division is made once per site, on Delta)
//   FsX  [V]           Re Tr of a site's four links, x 2^57
#pragma once
#include "lgf_aux.cuh"
#include "lgf_fx.cuh"

namespace lgf {

// x 2^57 from x 2^61, rounded to nearest
__device__ __forceinline__ fx to_sum(fx v) { return (v + 8) >> 4; }

// packed anti-Hermitian part of a link (rows w[0..5], row 2 w2) and its Re Tr
__device__ __forceinline__ void fx_ah(const cfx* w, const cfx* w2, cfx* a, fx& retr)
{
    a[0] = cfx{to_sum(w[1].re - w[3].re), to_sum(w[1].im + w[3].im)};
    a[1] = cfx{to_sum(w[2].re - w2[0].re), to_sum(w[2].im + w2[0].im)};
    a[2] = cfx{to_sum(w[5].re - w2[1].re), to_sum(w[5].im + w2[1].im)};
    const fx s0 = to_sum(w[0].im), s1 = to_sum(w[4].im), s2 = to_sum(w2[2].im);
    a[3] = cfx{2 * s0 - s1 - s2, 2 * s1 - s0 - s2};
    retr += to_sum(w[0].re) + to_sum(w[4].re) + to_sum(w2[2].re);
}

// Rows 0,1 of w = ga u gb^dag: A = rows of ga times u, then times gb^dag.  Each
// loads its operands' digits itself, so that u and gb are not held together.
// ua: rows 0,1 of u; u2: its row 2 is rebuilt here.
__device__ __forceinline__ void fx_link_gug(const cdig* ga, const cfx* u, const cdig* gb, cfx* w)
{
    cdig A[6];
    {
        cdig ud[9];
#pragma unroll
        for (int e = 0; e < 6; e++) ud[e] = digits(u[e]);
        cfx u2[3];
        fx_row2(ud, ud + 3, u2);
#pragma unroll
        for (int e = 0; e < 3; e++) ud[6 + e] = digits(u2[e]);
        cfx t[3];
#pragma unroll
        for (int i = 0; i < 2; i++) {
            fx_row_mul(ga + 3 * i, ud, t);
#pragma unroll
            for (int j = 0; j < 3; j++) A[3 * i + j] = digits(t[j]);
        }
    }
    fx_row_mul_dag(A, gb, w);
    fx_row_mul_dag(A + 3, gb, w + 3);
}

// G(x) <- g(x) G(x)
__device__ __forceinline__ void fx_gauge_accumulate(longlong2* __restrict__ G, int V, int s, const cdig* gx)
{
    cdig m[9];
#pragma unroll
    for (int e = 0; e < 6; e++) {
        const longlong2 v = G[(size_t)e * V + s];
        m[e] = digits(cfx{v.x, v.y});
    }
    cfx m2[3];
    fx_row2(m, m + 3, m2);
#pragma unroll
    for (int e = 0; e < 3; e++) m[6 + e] = digits(m2[e]);
#pragma unroll
    for (int i = 0; i < 2; i++) {
        cfx o[3];
        fx_row_mul(gx + 3 * i, m, o);
#pragma unroll
        for (int j = 0; j < 3; j++) stx(G + (size_t)(3 * i + j) * V + s, o[j]);
    }
}

// The update of one site: U'_mu(x) = g(x) U_mu(x) g^dag(x+mu) in place, the
// packed parts and Re Tr of the new links, G(x) <- g(x) G(x).
//
// Bound (32^4): 2600 mad.wide.s32 per site on a pipe of 63 per clock and SM
// (0.135 ms) and 1368 B/site of HBM traffic (0.21 ms).  One direction per pass of
// a rolled loop keeps the code in the instruction cache and the registers at 128
// (16 warps per SM).
static __global__ void __launch_bounds__(128, 4) k_update_fx(Lat d, longlong2* __restrict__ U,
                                                             longlong2* __restrict__ G,
                                                             const longlong2* __restrict__ g, Ctl* ctl,
                                                             longlong2* __restrict__ AH, fx* __restrict__ Fs)
{
    if (ld_flag(&ctl->phase_done)) return;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        ctl->iter += 1;
        if (ctl->phase == 0) ctl->iter_phase0 += 1;
    }
    const int V = d.V;
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= V) return;
    int c[4];
    site_coords(d, s, c);
    cdig gx[9];
#pragma unroll
    for (int e = 0; e < 9; e++) gx[e] = digits(ldx(g + (size_t)e * V + s));
    fx f = 0;
#pragma unroll 1
    for (int mu = 0; mu < 4; mu++) {
        const int cm = mu == 0 ? c[0] : mu == 1 ? c[1] : mu == 2 ? c[2] : c[3];
        const int sn = site_shift(d, s, cm, mu, +1);
        cfx u[6], w[6], w2[3];
#pragma unroll
        for (int e = 0; e < 6; e++) {
            const longlong2 v = U[(size_t)(mu * 6 + e) * V + s];
            u[e] = cfx{v.x, v.y};
        }
        cdig gn[9];
#pragma unroll
        for (int e = 0; e < 9; e++) gn[e] = digits(ldx(g + (size_t)e * V + sn));
        fx_link_gug(gx, u, gn, w);
        {
            cdig wd[6];
#pragma unroll
            for (int e = 0; e < 6; e++) {
                stx(U + (size_t)(mu * 6 + e) * V + s, w[e]);
                wd[e] = digits(w[e]);
            }
            fx_row2(wd, wd + 3, w2);
        }
        cfx a[4];
        fx_ah(w, w2, a, f);
#pragma unroll
        for (int k = 0; k < 4; k++) stx(AH + (size_t)(mu * 4 + k) * V + s, a[k]);
    }
    Fs[s] = f;
    if (G != nullptr) fx_gauge_accumulate(G, V, s, gx);
}

// Start of a loop: the links' rows 0,1 (and G's) on the grid, rounded to nearest,
// with their packed parts and Re Tr.
static __global__ void __launch_bounds__(128) k_fx_start(Lat d, const double2* __restrict__ U64,
                                                         const double2* __restrict__ G64, longlong2* __restrict__ U,
                                                         longlong2* __restrict__ G, longlong2* __restrict__ AH,
                                                         fx* __restrict__ Fs)
{
    const int V = d.V;
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= V) return;
    fx f = 0;
#pragma unroll 1
    for (int mu = 0; mu < 4; mu++) {
        cx<double> u[9];
        load_link<double>(U64, V, d.ne, mu, s, u);
        cfx w[6], w2[3], a[4];
        cdig wd[6];
#pragma unroll
        for (int e = 0; e < 6; e++) {
            w[e] = cfx{__double2ll_rn(u[e].re * 0x1p61), __double2ll_rn(u[e].im * 0x1p61)};
            wd[e] = digits(w[e]);
            stx(U + (size_t)(mu * 6 + e) * V + s, w[e]);
        }
        fx_row2(wd, wd + 3, w2);
        fx_ah(w, w2, a, f);
#pragma unroll
        for (int k = 0; k < 4; k++) stx(AH + (size_t)(mu * 4 + k) * V + s, a[k]);
    }
    Fs[s] = f;
    if (G != nullptr) {
#pragma unroll
        for (int e = 0; e < 6; e++) {
            const double2 v = G64[(size_t)e * V + s];
            stx(G + (size_t)e * V + s, cfx{__double2ll_rn(v.x * 0x1p61), __double2ll_rn(v.y * 0x1p61)});
        }
    }
}

// Start of the FP64 loop after the FP32 phase: the links rebuilt on the input's
// gauge orbit, U_mu(x) = Gs(x) U_in,mu(x) Gs^dag(x+mu), and G(x) <- Gs(x) G(x),
// straight onto the grid (Gs: [9][V], re-orthonormalised in FP64).
static __global__ void __launch_bounds__(128) k_fx_project(Lat d, const double2* __restrict__ U64,
                                                           const double2* __restrict__ G64,
                                                           const double2* __restrict__ Gs, longlong2* __restrict__ U,
                                                           longlong2* __restrict__ G, longlong2* __restrict__ AH,
                                                           fx* __restrict__ Fs, const Ctl* ctl)
{
    if (ld_flag(&ctl->nan_seen)) return;
    const int V = d.V;
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= V) return;
    int c[4];
    site_coords(d, s, c);
    bool bad = false;
    auto load_gs = [&](int site, cdig* m) {
#pragma unroll
        for (int e = 0; e < 9; e++) {
            const cx<double> v = ld<double>(Gs + (size_t)e * V + site);
            m[e] = digits(cfx{d2fx(v.re, &bad), d2fx(v.im, &bad)});
        }
    };
    cdig gx[9];
    load_gs(s, gx);
    fx f = 0;
#pragma unroll 1
    for (int mu = 0; mu < 4; mu++) {
        const int cm = mu == 0 ? c[0] : mu == 1 ? c[1] : mu == 2 ? c[2] : c[3];
        cfx u[6], w[6], w2[3], a[4];
        {
            cx<double> ud[9];
            load_link<double>(U64, V, d.ne, mu, s, ud);
#pragma unroll
            for (int e = 0; e < 6; e++) u[e] = cfx{d2fx(ud[e].re, &bad), d2fx(ud[e].im, &bad)};
        }
        cdig gn[9];
        load_gs(site_shift(d, s, cm, mu, +1), gn);
        fx_link_gug(gx, u, gn, w);
        cdig wd[6];
#pragma unroll
        for (int e = 0; e < 6; e++) {
            stx(U + (size_t)(mu * 6 + e) * V + s, w[e]);
            wd[e] = digits(w[e]);
        }
        fx_row2(wd, wd + 3, w2);
        fx_ah(w, w2, a, f);
#pragma unroll
        for (int k = 0; k < 4; k++) stx(AH + (size_t)(mu * 4 + k) * V + s, a[k]);
    }
    Fs[s] = f;
    if (G != nullptr) {
#pragma unroll
        for (int e = 0; e < 6; e++) {
            const double2 v = G64[(size_t)e * V + s];
            stx(G + (size_t)e * V + s, cfx{d2fx(v.x, &bad), d2fx(v.y, &bad)});
        }
        fx_gauge_accumulate(G, V, s, gx);
    }
    if (bad) const_cast<Ctl*>(ctl)->bad = 1;
}

// End of a loop: links and G back to FP64 in the context's form (NaN when an entry
// of g was not finite, as the links then are).  Nothing is written when no update
// was made (always: the start's links are not the stored ones, mixed mode), nor
// after a NaN in the FP32 phase.
static __global__ void __launch_bounds__(128) k_fx_finish(Lat d, const longlong2* __restrict__ U,
                                                          const longlong2* __restrict__ G,
                                                          double2* __restrict__ U64, double2* __restrict__ G64,
                                                          const Ctl* ctl, int always)
{
    const bool bad = ld_flag(&ctl->bad) != 0;
    if (ld_flag(&ctl->nan_seen) && !bad) return;
    if (!always && ld_flag(&ctl->iter) == 0) return;
    const int V = d.V;
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= V) return;
    const double nan = __hiloint2double(0x7ff80000, 0);
    auto back = [&](longlong2 v) {
        return bad ? mk<double>(nan, nan) : mk<double>(fx2d(v.x, kFxBits), fx2d(v.y, kFxBits));
    };
#pragma unroll 1
    for (int mu = 0; mu < 4; mu++) {
        cx<double> w[9];
#pragma unroll
        for (int e = 0; e < 6; e++) w[e] = back(__ldg(U + (size_t)(mu * 6 + e) * V + s));
        if (d.ne != 6) complete_row2(w, w + 6);
        store_link<double>(U64, V, d.ne, mu, s, w);
    }
    if (G != nullptr) {
#pragma unroll
        for (int e = 0; e < 6; e++) st<double>(G64 + (size_t)e * V + s, back(__ldg(G + (size_t)e * V + s)));
    }
}

// k_delta on the fixed-point parts: the stencil's 56 additions per site are integer
// (exact); Delta, theta and F in FP64 from there on.  Otherwise as k_delta.
template <bool FFT, int LMAX, typename TF>
__global__ void __launch_bounds__(kTileMaxThreads<double>, kTileMinBlocks<double, LMAX>) k_delta_fx(
    Lat d, const longlong2* __restrict__ AH, const fx* __restrict__ Fs, vec2_t<TF>* __restrict__ Fd,
    double* __restrict__ partials, Ctl* ctl, double2* hist)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    vec2_t<TF>* sm = reinterpret_cast<vec2_t<TF>*>(smem_raw);
    if (ld_flag(&ctl->phase_done)) return;
    const int P = d.P, V = d.V, Lx = d.L[0];
    const int plane = blockIdx.x;
    const int s0 = plane * P;
    const int z = plane % d.L[2], t = plane / d.L[2];
    const int rsx = plane_rsx(d), fs = plane_fs(d);
    double th = 0.0, fsum = 0.0;
#pragma unroll 2
    for (int xy = threadIdx.x; xy < P; xy += blockDim.x) {
        const int s = s0 + xy;
        const int y = (int)fdiv((unsigned)xy, d.dLx), x = xy - y * Lx;
        const int c[4] = {x, y, z, t};
        int sb[4];
#pragma unroll
        for (int mu = 0; mu < 4; mu++) sb[mu] = site_shift(d, s, c[mu], mu, -1);
        cfx a[16], b[16];
#pragma unroll
        for (int mu = 0; mu < 4; mu++)
#pragma unroll
            for (int k = 0; k < 4; k++) {
                a[4 * mu + k] = ldx(AH + (size_t)(mu * 4 + k) * V + sb[mu]);
                b[4 * mu + k] = ldx(AH + (size_t)(mu * 4 + k) * V + s);
            }
        fsum += fx2d(__ldg(Fs + s), kFxSum);
        cx<double> D[4];
#pragma unroll
        for (int k = 0; k < 4; k++) {
            fx re = 0, im = 0;
#pragma unroll
            for (int mu = 0; mu < 4; mu++) {
                re += a[4 * mu + k].re - b[4 * mu + k].re;
                im += a[4 * mu + k].im - b[4 * mu + k].im;
            }
            D[k] = mk<double>(fx2d(re, kFxSum), fx2d(im, kFxSum));
        }
        D[3] = D[3] * (2.0 / 3.0);
        th += theta_site(D);
        if (FFT) {
#pragma unroll
            for (int k = 0; k < 4; k++) st<TF>(sm + k * fs + y * rsx + x, to_tf<TF>(D[k]));
        } else {
#pragma unroll
            for (int k = 0; k < 4; k++) st<TF>(Fd + (size_t)k * V + s, to_tf<TF>(D[k]));
        }
    }
    reduce_theta_F(th, fsum, partials, ctl, hist, V);
    if (FFT) {
        __syncthreads();
        tile_x_lines<TF, false, LMAX>(d, sm);
        __syncthreads();
        plane_y_lines<TF, false, LMAX>(d, sm, fs, rsx, Fd + s0, V, Lx);
    }
}

// Whether every stored link is within 1e-3 of SU(3) (rows 0,1 orthonormal): the
// range the fixed-point products are bounded for.  *wide counts the others.
static __global__ void k_check_range(Lat d, const double2* __restrict__ U64, int* wide)
{
    const long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= 4L * d.V) return;
    const int mu = (int)(idx / d.V), s = (int)(idx - (long)mu * d.V);
    cx<double> u[9];
    load_link<double>(U64, d.V, d.ne, mu, s, u);
    cx<float> r[6];
#pragma unroll
    for (int e = 0; e < 6; e++) r[e] = mk<float>((float)u[e].re, (float)u[e].im);
    const float n0 = norm2(r[0]) + norm2(r[1]) + norm2(r[2]), n1 = norm2(r[3]) + norm2(r[4]) + norm2(r[5]);
    cx<float> ip = cmulc(r[3], r[0]);
    ip = cmacc(ip, r[4], r[1]);
    ip = cmacc(ip, r[5], r[2]);
    const bool ok = fabsf(n0 - 1.f) < 1e-3f && fabsf(n1 - 1.f) < 1e-3f && norm2(ip) < 1e-6f;
    if (!ok) *wide = 1;
}

}  // namespace lgf
