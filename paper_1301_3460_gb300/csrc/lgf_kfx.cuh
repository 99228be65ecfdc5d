// The FP64 iterations on 64-bit fixed point (lgf_fx.cuh): start and end of a
// loop, the update and the Delta stencil.  Arrays of a loop:
//   UX   [mu=4][6][V]  rows 0,1 of every link, x 2^61 in digits (whatever form the
//                      context stores its FP64 links in)
//   gX   [9][V]        g, x 2^62 in digits
//   AHX  [mu=4][4][V]  packed anti-Hermitian parts of the links, x 2^58; the
//                      fourth entry holds 2 Im w00 - Im w11 - Im w22 and 2 Im w11
//                      - Im w00 - Im w22 (3/2 of the packed traceless diagonal:
//                      the division is made once per site, on Delta)
//   FsX  [V]           Re Tr of a site's four links, x 2^58
// Values go to the coarser grid by an arithmetic shift (toward minus infinity):
// the mean error is the same for every link and cancels in Delta, which is made of
// differences.
#pragma once
#include "lgf_aux.cuh"
#include "lgf_fx.cuh"

namespace lgf {

__device__ __forceinline__ fx to_sum(fx v) { return v >> (kFxBits - kFxSum); }

// packed anti-Hermitian part of a link and its Re Tr: rows w[0..5] (2^-61), row 2
// rebuilt from their digits (at 2^-58, where it needs no shift)
__device__ __forceinline__ void fx_ah(const cfx* w, const cdig* wd, cfx* a, fx& retr)
{
    cfx w2[3];
#pragma unroll
    for (int j = 0; j < 3; j++) w2[j] = fx_row2<0>(wd, wd + 3, j);
    a[0] = cfx{to_sum(w[1].re - w[3].re), to_sum(w[1].im + w[3].im)};
    a[1] = cfx{to_sum(w[2].re) - w2[0].re, to_sum(w[2].im) + w2[0].im};
    a[2] = cfx{to_sum(w[5].re) - w2[1].re, to_sum(w[5].im) + w2[1].im};
    const fx s0 = to_sum(w[0].im), s1 = to_sum(w[4].im), t = s0 + s1 + w2[2].im;
    a[3] = cfx{3 * s0 - t, 3 * s1 - t};
    retr += to_sum(w[0].re + w[4].re) + w2[2].re;
}

// Row 2 of a link from the digits of its rows 0,1 and its packed part: the
// off-diagonal entries of the part are w02 - conj(w20) and w12 - conj(w21), its
// diagonal gives Im w22, so only Re w22 is multiplied out (60 of 72 integer
// products less, for 48 bytes read; the same values as fx_ah's row 2).
__device__ __forceinline__ void fx_row2_from_part(const cdig* r, const longlong2* part, cfx* r2)
{
    const fx w02r = to_sum(value(r[2].re)), w02i = to_sum(value(r[2].im));
    const fx w12r = to_sum(value(r[5].re)), w12i = to_sum(value(r[5].im));
    const fx s0 = to_sum(value(r[0].im)), s1 = to_sum(value(r[4].im));
    r2[0] = cfx{w02r - part[0].x, part[0].y - w02i};
    r2[1] = cfx{w12r - part[1].x, part[1].y - w12i};
    // part[2].x = 3 s0 - (s0 + s1 + Im w22)
    facc p = fmul<0>(r[0].re, r[4].re), n = fmul<0>(r[0].im, r[4].im);
    fmac(p, r[1].im, r[3].im);
    fmac(n, r[1].re, r[3].re);
    r2[2] = cfx{fval<0>(fsub(p, n)), 2 * s0 - s1 - part[2].x};
#pragma unroll
    for (int j = 0; j < 3; j++) r2[j] = cfx{r2[j].re << (kFxBits - kFxSum), r2[j].im << (kFxBits - kFxSum)};
}

// Rows 0,1 of w = ga u gb^dag: A = rows 0,1 of ga times u (at 2^-59, unshifted), then
// times gb^dag.  u: digits of rows 0,1; u2: row 2; gb: digits of all three rows.
__device__ __forceinline__ void fx_link_gug(const cdig3* ga, const cdig* u, const cfx* u2, const cdig* gb, cfx* w)
{
    cdig3 A[6];
    {
        cdig3 ud[9];
#pragma unroll
        for (int e = 0; e < 6; e++) ud[e] = with_sum(u[e]);
#pragma unroll
        for (int j = 0; j < 3; j++) ud[6 + j] = with_sum(u2[j]);
#pragma unroll
        for (int j = 0; j < 3; j++) {
            A[j] = with_diff(fx_mul<0>(ga, ud, j));
            A[3 + j] = with_diff(fx_mul<0>(ga + 3, ud, j));
        }
    }
    cdig3 b[9];
#pragma unroll
    for (int e = 0; e < 9; e++) b[e] = with_sum(gb[e]);
#pragma unroll
    for (int j = 0; j < 3; j++) {
        w[j] = fx_mul_dag<4>(A, b, j);
        w[3 + j] = fx_mul_dag<4>(A + 3, b, j);
    }
}

// stores link (mu, s) and its packed part
__device__ __forceinline__ void fx_store_link(longlong2* __restrict__ U, longlong2* __restrict__ AH, int V, int mu,
                                              int s, const cfx* w, fx& f)
{
    cdig wd[6];
#pragma unroll
    for (int e = 0; e < 6; e++) {
        wd[e] = digits(w[e]);
        std_(U + (size_t)(mu * 6 + e) * V + s, wd[e]);
    }
    cfx a[4];
    fx_ah(w, wd, a, f);
#pragma unroll
    for (int k = 0; k < 4; k++) stx(AH + (size_t)(mu * 4 + k) * V + s, a[k]);
}

// The update of one site: U'_mu(x) = g(x) U_mu(x) g^dag(x+mu) in place, the
// packed parts and Re Tr of the new links, G(x) <- g(x) G(x).  G stays in FP64: its
// 96 operations per site run on the FP64 pipe beside the integer products.
//
// Bound (32^4): 1630 mad.wide.s32 per site (24 per clock and SM with distinct
// operands: 0.23 ms) and 1560 B/site of HBM traffic (0.24 ms).  One direction per
// pass of a rolled loop keeps the code in the instruction cache.
__device__ __forceinline__ void fx_update_site(const Lat& d, longlong2* __restrict__ U, double2* __restrict__ G,
                                               const longlong2* __restrict__ g, longlong2* __restrict__ AH,
                                               fx* __restrict__ Fs, int s)
{
    const int V = d.V;
    int c[4];
    site_coords(d, s, c);
    cdig3 gx[6];
#pragma unroll
    for (int e = 0; e < 6; e++) gx[e] = with_sum(ldd(g + (size_t)e * V + s));
    fx f = 0;
#pragma unroll 1
    for (int mu = 0; mu < 4; mu++) {
        const int cm = mu == 0 ? c[0] : mu == 1 ? c[1] : mu == 2 ? c[2] : c[3];
        const int sn = site_shift(d, s, cm, mu, +1);
        cdig u[6], gn[9];
        longlong2 part[3];
#pragma unroll
        for (int e = 0; e < 6; e++) u[e] = unpack(U[(size_t)(mu * 6 + e) * V + s]);
#pragma unroll
        for (int k = 0; k < 3; k++) part[k] = AH[(size_t)(mu * 4 + 1 + k) * V + s];
#pragma unroll
        for (int e = 0; e < 9; e++) gn[e] = ldd(g + (size_t)e * V + sn);
        cfx u2[3], w[6];
        fx_row2_from_part(u, part, u2);
        fx_link_gug(gx, u, u2, gn, w);
        fx_store_link(U, AH, V, mu, s, w, f);
    }
    Fs[s] = f;
    if (G != nullptr) {
        cx<double> gd[6];
#pragma unroll
        for (int e = 0; e < 6; e++) gd[e] = mk<double>(fx2d(value(gx[e].re), kFxG), fx2d(value(gx[e].im), kFxG));
        gauge_accumulate<double>(G, V, s, gd);
    }
}

static __global__ void __launch_bounds__(64, 6) k_update_fx(Lat d, longlong2* __restrict__ U,
                                                            double2* __restrict__ G,
                                                             const longlong2* __restrict__ g, Ctl* ctl,
                                                             longlong2* __restrict__ AH, fx* __restrict__ Fs)
{
    if (ld_flag(&ctl->phase_done)) return;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        ctl->iter += 1;
        if (ctl->phase == 0) ctl->iter_phase0 += 1;
    }
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s < d.V) fx_update_site(d, U, G, g, AH, Fs, s);
}

// magnitude exponents of the integer transform's fields (lgf_fxt.cuh)
constexpr int kExpNone = -(1 << 28);
struct FxExp {
    int amax1;  // over the planes, after the Delta kernel (reset at the start of a loop and by the g builder)
    int amax2;  // over the pencils, after the accelerator (reset by the Delta kernel)
};

// Start of a loop: the links' rows 0,1 on the grid, rounded to nearest, with their
// packed parts and Re Tr.
static __global__ void __launch_bounds__(128) k_fx_start(Lat d, const double2* __restrict__ U64,
                                                         longlong2* __restrict__ U, longlong2* __restrict__ AH,
                                                         fx* __restrict__ Fs, FxExp* fe)
{
    const int V = d.V;
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s == 0) fe->amax1 = kExpNone;
    if (s >= V) return;
    fx f = 0;
#pragma unroll 1
    for (int mu = 0; mu < 4; mu++) {
        cx<double> u[9];
        load_link<double>(U64, V, d.ne, mu, s, u);
        cfx w[6];
#pragma unroll
        for (int e = 0; e < 6; e++) w[e] = cfx{__double2ll_rn(u[e].re * 0x1p61), __double2ll_rn(u[e].im * 0x1p61)};
        fx_store_link(U, AH, V, mu, s, w, f);
    }
    Fs[s] = f;
}

// Start of the FP64 loop after the FP32 phase: the links rebuilt on the input's
// gauge orbit, U_mu(x) = Gs(x) U_in,mu(x) Gs^dag(x+mu), and G(x) <- Gs(x) G(x),
// straight onto the grid (Gs: [9][V], re-orthonormalised in FP64).
static __global__ void __launch_bounds__(128) k_fx_project(Lat d, const double2* __restrict__ U64,
                                                           double2* __restrict__ G, const double2* __restrict__ Gs,
                                                           longlong2* __restrict__ U, longlong2* __restrict__ AH,
                                                           fx* __restrict__ Fs, FxExp* fe, const Ctl* ctl)
{
    if (ld_flag(&ctl->nan_seen)) return;
    const int V = d.V;
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s == 0) fe->amax1 = kExpNone;
    if (s >= V) return;
    int c[4];
    site_coords(d, s, c);
    bool bad = false;
    auto load_gs = [&](int site, int e) {
        const cx<double> v = ld<double>(Gs + (size_t)e * V + site);
        return digits(cfx{d2fx<kFxG>(v.re, &bad), d2fx<kFxG>(v.im, &bad)});
    };
    cdig3 gx[6];
#pragma unroll
    for (int e = 0; e < 6; e++) gx[e] = with_sum(load_gs(s, e));
    fx f = 0;
#pragma unroll 1
    for (int mu = 0; mu < 4; mu++) {
        const int cm = mu == 0 ? c[0] : mu == 1 ? c[1] : mu == 2 ? c[2] : c[3];
        cdig u[6], gn[9];
        {
            cx<double> ud[9];
            load_link<double>(U64, V, d.ne, mu, s, ud);
#pragma unroll
            for (int e = 0; e < 6; e++)
                u[e] = digits(cfx{d2fx<kFxBits>(ud[e].re, &bad), d2fx<kFxBits>(ud[e].im, &bad)});
        }
        const int sn = site_shift(d, s, cm, mu, +1);
#pragma unroll
        for (int e = 0; e < 9; e++) gn[e] = load_gs(sn, e);
        cfx u2[3], w[6];
#pragma unroll
        for (int j = 0; j < 3; j++) u2[j] = fx_row2<3>(u, u + 3, j);
        fx_link_gug(gx, u, u2, gn, w);
        fx_store_link(U, AH, V, mu, s, w, f);
    }
    Fs[s] = f;
    if (G != nullptr) {
        cx<double> gd[6];
#pragma unroll
        for (int e = 0; e < 6; e++) gd[e] = ld<double>(Gs + (size_t)e * V + s);
        gauge_accumulate<double>(G, V, s, gd);
    }
    if (bad) const_cast<Ctl*>(ctl)->bad = 1;
}

// End of a loop: links back to FP64 in the context's form (links and G NaN when an
// entry of g was not finite).  Nothing is written when no update was made (always:
// the start's links are not the stored ones, mixed mode), nor after a NaN in the
// FP32 phase.
static __global__ void __launch_bounds__(128) k_fx_finish(Lat d, const longlong2* __restrict__ U,
                                                          double2* __restrict__ U64, double2* __restrict__ G,
                                                          const Ctl* ctl, int always)
{
    const bool bad = ld_flag(&ctl->bad) != 0;
    if (ld_flag(&ctl->nan_seen) && !bad) return;
    if (!always && ld_flag(&ctl->iter) == 0) return;
    const int V = d.V;
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= V) return;
    const cx<double> nan = mk<double>(__hiloint2double(0x7ff80000, 0), __hiloint2double(0x7ff80000, 0));
#pragma unroll 1
    for (int mu = 0; mu < 4; mu++) {
        cx<double> w[9];
#pragma unroll
        for (int e = 0; e < 6; e++) {
            const cdig v = ldd(U + (size_t)(mu * 6 + e) * V + s);
            w[e] = bad ? nan : mk<double>(fx2d(value(v.re), kFxBits), fx2d(value(v.im), kFxBits));
        }
        if (d.ne != 6) complete_row2(w, w + 6);
        store_link<double>(U64, V, d.ne, mu, s, w);
    }
    if (bad && G != nullptr)
        for (int e = 0; e < 6; e++) st<double>(G + (size_t)e * V + s, nan);
}

// Delta of the sites of one xy-plane from the fixed-point parts: the stencil's 56
// additions per site are integer (exact); theta and F accumulate in FP64.
// out(xy, x, y, raw, D): the packed sums x 2^58 (field 3 times 3/2) and Delta.
template <typename OUT>
__device__ __forceinline__ void fx_delta_plane(const Lat& d, const longlong2* __restrict__ AH,
                                               const fx* __restrict__ Fs, int plane, double& th, double& fsum, OUT out)
{
    const int P = d.P, V = d.V, Lx = d.L[0];
    const int s0 = plane * P;
    const int z = plane % d.L[2], t = plane / d.L[2];
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
        cfx raw[4];
        cx<double> D[4];
#pragma unroll
        for (int k = 0; k < 4; k++) {
            raw[k] = cfx{0, 0};
#pragma unroll
            for (int mu = 0; mu < 4; mu++) raw[k] = raw[k] + a[4 * mu + k] - b[4 * mu + k];
            D[k] = mk<double>(fx2d(raw[k].re, kFxSum), fx2d(raw[k].im, kFxSum));
        }
        D[3] = D[3] * (2.0 / 3.0);
        th += theta_site(D);
        out(xy, x, y, raw, D);
    }
}

// k_delta on the fixed-point parts, with Delta itself (FFT false) or its forward x,y
// transform in TF.
template <bool FFT, int LMAX, typename TF>
__global__ void __launch_bounds__(kTileMaxThreads<double>, kTileMinBlocks<double, LMAX>) k_delta_fx(
    Lat d, const longlong2* __restrict__ AH, const fx* __restrict__ Fs, vec2_t<TF>* __restrict__ Fd,
    double* __restrict__ partials, Ctl* ctl, double2* hist)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    vec2_t<TF>* sm = reinterpret_cast<vec2_t<TF>*>(smem_raw);
    if (ld_flag(&ctl->phase_done)) return;
    const int V = d.V, Lx = d.L[0], s0 = blockIdx.x * d.P;
    const int rsx = plane_rsx(d), fs = plane_fs(d);
    double th = 0.0, fsum = 0.0;
    fx_delta_plane(d, AH, Fs, blockIdx.x, th, fsum, [&](int xy, int x, int y, const cfx*, const cx<double>* D) {
#pragma unroll
        for (int k = 0; k < 4; k++) {
            if (FFT) st<TF>(sm + k * fs + y * rsx + x, to_tf<TF>(D[k]));
            else st<TF>(Fd + (size_t)k * V + s0 + xy, to_tf<TF>(D[k]));
        }
    });
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
