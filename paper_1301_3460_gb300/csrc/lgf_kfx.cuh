// The FP64 iterations on 64-bit fixed point (lgf_fx.cuh): start and end of a
// loop, the update and the Delta stencil.  Arrays of a loop:
//   UX   [mu=4][nx][V] rows 0,1 of every link, x 2^61, in the first six planes of
//                      each direction (whatever form the context stores its FP64 links
//                      in).  Without an FP32 phase they take the FP64 links' place while
//                      the loop runs (nx is 9 over 18-real links, else 6), with one the
//                      idle FP32 links' place: no memory of their own
//   GX   [6][V]        rows 0,1 of G, x 2^61 (null: not tracked), likewise
//   gX   [9][V]        g, x 2^62
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

// Row 2 of a link from its rows 0,1 (w, digits r) and its packed part: the
// off-diagonal entries of the part are w02 - conj(w20) and w12 - conj(w21), its
// diagonal gives Im w22, so only Re w22 is multiplied out (60 of 72 integer
// products less, for 48 bytes read; the same values as fx_ah's row 2).
__device__ __forceinline__ void fx_row2_from_part(const cfx* w, const cdig3* r, const longlong2* part, cfx* r2)
{
    const fx w02r = to_sum(w[2].re), w02i = to_sum(w[2].im);
    const fx w12r = to_sum(w[5].re), w12i = to_sum(w[5].im);
    const fx s0 = to_sum(w[0].im), s1 = to_sum(w[4].im);
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

// A = rows 0,1 of ga times u (at 2^-59, unshifted), kept with their differences for the
// product with gb^dag
__device__ __forceinline__ void fx_left(const cdig3* ga, const cdig3* ud, cdig3* A)
{
#pragma unroll
    for (int j = 0; j < 3; j++) {
        A[j] = with_diff(fx_mul<0>(ga, ud, j));
        A[3 + j] = with_diff(fx_mul<0>(ga + 3, ud, j));
    }
}
// rows 0,1 of w = A gb^dag; gb(e): entry e of gb
template <typename GB> __device__ __forceinline__ void fx_right(const cdig3* A, GB gb, cfx* w)
{
#pragma unroll
    for (int j = 0; j < 3; j++) {
        cdig3 b[3];
#pragma unroll
        for (int k = 0; k < 3; k++) b[k] = with_sum(gb(3 * j + k));
        w[j] = fx_mul_dag<4>(A, b);
        w[3 + j] = fx_mul_dag<4>(A + 3, b);
    }
}

// stores link (mu, s) and its packed part
__device__ __forceinline__ void fx_store_link(longlong2* __restrict__ U, longlong2* __restrict__ AH, int V, int nx, int mu,
                                              int s, const cfx* w, fx& f)
{
    cdig wd[6];
#pragma unroll
    for (int e = 0; e < 6; e++) {
        wd[e] = digits(w[e]);
        stx(U + (size_t)(mu * nx + e) * V + s, w[e]);
    }
    cfx a[4];
    fx_ah(w, wd, a, f);
#pragma unroll
    for (int k = 0; k < 4; k++) stx(AH + (size_t)(mu * 4 + k) * V + s, a[k]);
}

// G(x) <- g(x) G(x): rows 0,1 (m on entry), G's row 2 rebuilt
__device__ __forceinline__ void fx_gauge_accumulate(longlong2* __restrict__ G, int V, int s, const cdig3* gx,
                                                    const cfx* m)
{
    cdig3 md[9];
#pragma unroll
    for (int e = 0; e < 6; e++) md[e] = with_sum(m[e]);
#pragma unroll
    for (int j = 0; j < 3; j++) md[6 + j] = with_sum(fx_row2<3>(md, md + 3, j));
#pragma unroll
    for (int i = 0; i < 2; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) stx(G + (size_t)(3 * i + j) * V + s, fx_mul<2>(gx + 3 * i, md, j));
}

// 16 bytes to the thread's own slot in shared memory, past L1 (streamed data) or
// through it (g, read by up to five sites)
template <bool L1> __device__ __forceinline__ void cp_async16(longlong2* dst, const longlong2* src)
{
    const unsigned a = (unsigned)__cvta_generic_to_shared(dst);
    if (L1) asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(a), "l"(src) : "memory");
    else asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(a), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// all but the newest group of this thread's copies have arrived
__device__ __forceinline__ void cp_async_wait1() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }

// The update of every site, one thread each: U'_mu(x) = g(x) U_mu(x) g^dag(x+mu) in
// place, the packed parts and Re Tr of the new links, G(x) <- g(x) G(x).
//
// Bound: 1632 (+ 234 with G) mad.wide.s32 per site, which issue at 24 to 32 per clock
// and SM with distinct operands (32^4: 0.21 to 0.28 ms), and 1560 B/site of HBM
// traffic (0.24 ms).  A thread holds some 120 registers, so 16 warps per SM: too few to
// wait out the loads.  Each direction's inputs are therefore copied to slots in shared
// memory of the thread's own (no barrier) one direction ahead: the link and its part as
// soon as the current ones are in registers, g(x+mu) as soon as it has been used; g(x)
// waits in shared memory too.  32^4, with G: 1630 us in FP64 (924 operations per site at
// 2 per clock and SM), 406 us on integers with loads where they are used, 315 us like
// this (77% of the HBM rate); without G 357 and 281 us.  G in FP64 beside the integer
// products is slower (441 against 406 us): it comes at the end of every thread.
// NX: the links' nx as a constant (as an argument it costs 0.7%: 1558 -> 1571 us at 48^4).
constexpr int kUpdThreads = 128;
template <int NX>
__global__ void __launch_bounds__(kUpdThreads, 4) k_update_fx(Lat d, longlong2* __restrict__ U, longlong2* __restrict__ G,
                                                              const longlong2* __restrict__ g, Ctl* ctl,
                                                              longlong2* __restrict__ AH, fx* __restrict__ Fs)
{
    __shared__ longlong2 slots[24 * kUpdThreads];  // per thread: link and part (9), g(x+mu) (9), rows 0,1 of g(x) (6)
    constexpr int NT = kUpdThreads;
    if (ld_flag(&ctl->phase_done)) return;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        ctl->iter += 1;
        if (ctl->phase == 0) ctl->iter_phase0 += 1;
    }
    const int V = d.V;
    const int s = blockIdx.x * NT + threadIdx.x;
    if (s >= V) return;
    longlong2 *su = slots + threadIdx.x, *sn = su + 9 * NT, *sx = sn + 9 * NT;
    int nb[4];
    {
        int c[4];
        site_coords(d, s, c);
#pragma unroll
        for (int mu = 0; mu < 4; mu++) nb[mu] = site_shift(d, s, c[mu], mu, +1);
    }
    auto fetch_u = [&](int mu) {
#pragma unroll
        for (int e = 0; e < 6; e++) cp_async16<false>(su + e * NT, U + (size_t)(mu * NX + e) * V + s);
#pragma unroll
        for (int k = 0; k < 3; k++) cp_async16<false>(su + (6 + k) * NT, AH + (size_t)(mu * 4 + 1 + k) * V + s);
    };
    auto fetch_g = [&](int site) {
#pragma unroll
        for (int e = 0; e < 9; e++) cp_async16<true>(sn + e * NT, g + (size_t)e * V + site);
    };
    fetch_u(0);
    cp_async_commit();
    fetch_g(nb[0]);
    cp_async_commit();
#pragma unroll
    for (int e = 0; e < 6; e++) sx[e * NT] = __ldg(g + (size_t)e * V + s);
    auto load_gx = [&](cdig3* gx) {
#pragma unroll
        for (int e = 0; e < 6; e++) gx[e] = with_sum(ldv<fx>(sx + e * NT));
    };
    fx f = 0;
#pragma unroll 1
    for (int mu = 0; mu < 4; mu++) {
        cfx u[9], w[6];
        cdig3 A[6];
        cp_async_wait1();
        {
            cdig3 ud[9];
            longlong2 part[3];
#pragma unroll
            for (int e = 0; e < 6; e++) u[e] = ldv<fx>(su + e * NT);
#pragma unroll
            for (int k = 0; k < 3; k++) part[k] = su[(6 + k) * NT];
#pragma unroll
            for (int e = 0; e < 6; e++) ud[e] = with_sum(u[e]);
            fx_row2_from_part(u, ud, part, u + 6);
            // the slots are free: the next direction's link, G after the last one
            if (mu < 3) {
                fetch_u(mu + 1);
            } else if (G != nullptr) {
#pragma unroll
                for (int e = 0; e < 6; e++) cp_async16<false>(su + e * NT, G + (size_t)e * V + s);
            }
            cp_async_commit();
#pragma unroll
            for (int e = 6; e < 9; e++) ud[e] = with_sum(u[e]);
            cdig3 gx[6];
            load_gx(gx);
            fx_left(gx, ud, A);
        }
        cp_async_wait1();
        fx_right(A, [&](int e) { return ldv<fx>(sn + e * NT); }, w);
        if (mu < 3) fetch_g(mu == 0 ? nb[1] : mu == 1 ? nb[2] : nb[3]);
        cp_async_commit();
        fx_store_link(U, AH, V, NX, mu, s, w, f);
    }
    Fs[s] = f;
    if (G != nullptr) {
        cp_async_wait1();
        cdig3 gx[6];
        cfx m[6];
        load_gx(gx);
#pragma unroll
        for (int e = 0; e < 6; e++) m[e] = ldv<fx>(su + e * NT);
        fx_gauge_accumulate(G, V, s, gx, m);
    }
}

// The same with a thread per link, a warp per direction of 32 sites and a fifth warp for
// G: for lattices that leave most of the chip idle with a thread per site, whose four
// links then follow one another (8^4: 14 us a launch against 9).
constexpr int kUpdSmallThreads = 160;
template <int NX>
__global__ void __launch_bounds__(kUpdSmallThreads, 3) k_update_fx_small(
    Lat d, longlong2* __restrict__ U, longlong2* __restrict__ G, const longlong2* __restrict__ g, Ctl* ctl,
    longlong2* __restrict__ AH, fx* __restrict__ Fs)
{
    __shared__ fx retr[4][32];
    if (ld_flag(&ctl->phase_done)) return;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        ctl->iter += 1;
        if (ctl->phase == 0) ctl->iter_phase0 += 1;
    }
    const int V = d.V, mu = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int s = blockIdx.x * 32 + lane;
    if (s < V) {
        cdig3 gx[6];
#pragma unroll
        for (int e = 0; e < 6; e++) gx[e] = with_sum(ldx(g + (size_t)e * V + s));
        if (mu < 4) {
            int c[4];
            site_coords(d, s, c);
            const int sn = site_shift(d, s, mu == 0 ? c[0] : mu == 1 ? c[1] : mu == 2 ? c[2] : c[3], mu, +1);
            cfx u[9], w[6], gn[9];
            longlong2 part[3];
#pragma unroll
            for (int e = 0; e < 6; e++) u[e] = ldv<fx>(U + (size_t)(mu * NX + e) * V + s);
#pragma unroll
            for (int k = 0; k < 3; k++) part[k] = AH[(size_t)(mu * 4 + 1 + k) * V + s];
#pragma unroll
            for (int e = 0; e < 9; e++) gn[e] = ldx(g + (size_t)e * V + sn);
            cdig3 A[6];
            {
                cdig3 ud[9];
#pragma unroll
                for (int e = 0; e < 6; e++) ud[e] = with_sum(u[e]);
                fx_row2_from_part(u, ud, part, u + 6);
#pragma unroll
                for (int e = 6; e < 9; e++) ud[e] = with_sum(u[e]);
                fx_left(gx, ud, A);
            }
            fx_right(A, [&](int e) { return gn[e]; }, w);
            fx f = 0;
            fx_store_link(U, AH, V, NX, mu, s, w, f);
            retr[mu][lane] = f;
        } else if (G != nullptr) {
            cfx m[6];
#pragma unroll
            for (int e = 0; e < 6; e++) m[e] = ldv<fx>(G + (size_t)e * V + s);
            fx_gauge_accumulate(G, V, s, gx, m);
        }
    }
    __syncthreads();
    if (mu == 0 && s < V) Fs[s] = retr[0][lane] + retr[1][lane] + retr[2][lane] + retr[3][lane];
}

// magnitude exponents of the integer transform's four fields (lgf_fxt.cuh)
constexpr int kExpNone = -(1 << 28);
struct __align__(16) FxExp {
    int amax1[4];  // over the planes, after the Delta kernel (reset at the start of a loop and by the g builder)
    int amax2[4];  // over the pencils, after the accelerator (reset by the Delta kernel)
    int bad;       // a field of FP64 values was not finite (k_xyfwd_fxt; reset before it)
    int pad[3];
};

// An FP64 link's rows 0,1 on the grid, rounded to nearest.  U64 may be the place that the
// fixed-point links go to, so it is read as integers (no read-only loads).
__device__ __forceinline__ void fx_rows_of_link(const longlong2* U64, int V, int ne, int mu, int s, cfx* w)
{
    const longlong2* p = U64 + (size_t)mu * ne * V + s;
    auto get = [&](int e) {
        const longlong2 v = p[(size_t)e * V];
        return mk<double>(__longlong_as_double(v.x), __longlong_as_double(v.y));
    };
    cx<double> u[9];
    if (ne == 4) {
        const cx<double> th = get(3);
        rebuild8<double>(get(0), get(1), get(2), th.re, th.im, u);
    } else {
#pragma unroll
        for (int e = 0; e < 6; e++) u[e] = get(e);
    }
#pragma unroll
    for (int e = 0; e < 6; e++) w[e] = cfx{d2fx_rn<kFxBits>(u[e].re), d2fx_rn<kFxBits>(u[e].im)};
}

// Start of a loop: the packed parts and Re Tr of the links on the grid.  The links stay what
// they are until there is an update to make (k_fx_enter).  U (may be null): a place of its
// own for the links on the grid.
static __global__ void __launch_bounds__(128) k_fx_start(Lat d, const longlong2* __restrict__ U64,
                                                         longlong2* __restrict__ U, longlong2* __restrict__ AH,
                                                         fx* __restrict__ Fs, FxExp* fe)
{
    const int V = d.V;
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s < 4) fe->amax1[s] = kExpNone;
    if (s >= V) return;
    fx f = 0;
#pragma unroll 1
    for (int mu = 0; mu < 4; mu++) {
        cfx w[6], a[4];
        cdig wd[6];
        fx_rows_of_link(U64, V, d.ne, mu, s, w);
#pragma unroll
        for (int e = 0; e < 6; e++) wd[e] = digits(w[e]);
        if (U != nullptr) {
#pragma unroll
            for (int e = 0; e < 6; e++) stx(U + (size_t)(mu * d.nx + e) * V + s, w[e]);
        }
        fx_ah(w, wd, a, f);
#pragma unroll
        for (int k = 0; k < 4; k++) stx(AH + (size_t)(mu * 4 + k) * V + s, a[k]);
    }
    Fs[s] = f;
}

// Before the first update: links and G to their fixed-point form, which may lie where the
// FP64 ones do (nx >= ne: from the last direction down, no link is overwritten before it is
// read, all by the site's own thread).  When the loop makes no update the stored links
// stay as they are.
static __global__ void __launch_bounds__(128) k_fx_enter(Lat d, const longlong2* U64, const longlong2* G64, longlong2* U,
                                                         longlong2* G, Ctl* ctl)
{
    if (ld_flag(&ctl->phase_done)) return;
    if (blockIdx.x == 0 && threadIdx.x == 0) ctl->fixed_form = 1;
    const int V = d.V;
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= V) return;
#pragma unroll 1
    for (int mu = 3; mu >= 0; mu--) {
        cfx w[6];
        fx_rows_of_link(U64, V, d.ne, mu, s, w);
#pragma unroll
        for (int e = 0; e < 6; e++) stx(U + (size_t)(mu * d.nx + e) * V + s, w[e]);
    }
    if (G != nullptr) {
#pragma unroll
        for (int e = 0; e < 6; e++) {
            const longlong2 v = G64[(size_t)e * V + s];
            stx(G + (size_t)e * V + s,
                cfx{d2fx_rn<kFxBits>(__longlong_as_double(v.x)), d2fx_rn<kFxBits>(__longlong_as_double(v.y))});
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
                                                           fx* __restrict__ Fs, FxExp* fe, const Ctl* ctl)
{
    if (ld_flag(&ctl->nan_seen)) return;
    const int V = d.V;
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s == 0) const_cast<Ctl*>(ctl)->fixed_form = 1;
    if (s < 4) fe->amax1[s] = kExpNone;
    if (s >= V) return;
    int c[4];
    site_coords(d, s, c);
    bool bad = false;
    auto load_gs = [&](int site, int e) {
        const cx<double> v = ld<double>(Gs + (size_t)e * V + site);
        return cfx{d2fx<kFxG>(v.re, &bad), d2fx<kFxG>(v.im, &bad)};
    };
    cdig3 gx[6];
#pragma unroll
    for (int e = 0; e < 6; e++) gx[e] = with_sum(load_gs(s, e));
    fx f = 0;
#pragma unroll 1
    for (int mu = 0; mu < 4; mu++) {
        const int cm = mu == 0 ? c[0] : mu == 1 ? c[1] : mu == 2 ? c[2] : c[3];
        const int sn = site_shift(d, s, cm, mu, +1);
        cfx w[6];
        cdig3 A[6];
        {
            cx<double> u[9];
            cdig3 ud[9];
            load_link<double>(U64, V, d.ne, mu, s, u);
#pragma unroll
            for (int e = 0; e < 6; e++) ud[e] = with_sum(cfx{d2fx<kFxBits>(u[e].re, &bad), d2fx<kFxBits>(u[e].im, &bad)});
#pragma unroll
            for (int j = 0; j < 3; j++) ud[6 + j] = with_sum(fx_row2<3>(ud, ud + 3, j));
            fx_left(gx, ud, A);
        }
        fx_right(A, [&](int e) { return load_gs(sn, e); }, w);
        fx_store_link(U, AH, V, d.nx, mu, s, w, f);
    }
    Fs[s] = f;
    if (G != nullptr) {
        cfx m[6];
#pragma unroll
        for (int e = 0; e < 6; e++) {
            const double2 v = G64[(size_t)e * V + s];
            m[e] = cfx{d2fx<kFxBits>(v.x, &bad), d2fx<kFxBits>(v.y, &bad)};
        }
        fx_gauge_accumulate(G, V, s, gx, m);
    }
    if (bad) const_cast<Ctl*>(ctl)->bad = 1;
}

// End of a loop that took the links to their fixed-point form: links and G back to FP64 in
// the context's form, which may lie in the same place (ne <= nx: from the first direction
// up), NaN when an entry of g was not finite.
static __global__ void __launch_bounds__(128) k_fx_finish(Lat d, const longlong2* U, const longlong2* G, double2* U64,
                                                          double2* G64, const Ctl* ctl)
{
    if (!ld_flag(&ctl->fixed_form)) return;
    const bool bad = ld_flag(&ctl->bad) != 0;
    const int V = d.V;
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= V) return;
    const cx<double> nan = mk<double>(__hiloint2double(0x7ff80000, 0), __hiloint2double(0x7ff80000, 0));
    auto back = [&](cfx v) { return bad ? nan : mk<double>(fx2d(v.re, kFxBits), fx2d(v.im, kFxBits)); };
#pragma unroll 1
    for (int mu = 0; mu < 4; mu++) {
        cx<double> w[9];
#pragma unroll
        for (int e = 0; e < 6; e++) w[e] = back(ldv<fx>(U + (size_t)(mu * d.nx + e) * V + s));
        if (d.ne != 6) complete_row2(w, w + 6);
        // the loads above come first whatever types the two views of the place have
        asm volatile("" ::: "memory");
        store_link<double>(U64, V, d.ne, mu, s, w);
        asm volatile("" ::: "memory");
    }
    if (G != nullptr) {
        cx<double> m[6];
#pragma unroll
        for (int e = 0; e < 6; e++) m[e] = back(ldv<fx>(G + (size_t)e * V + s));
        asm volatile("" ::: "memory");
#pragma unroll
        for (int e = 0; e < 6; e++) st<double>(G64 + (size_t)e * V + s, m[e]);
    }
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
    double* __restrict__ partials, Ctl* ctl, double2* hist, cudaGraphConditionalHandle h)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    vec2_t<TF>* sm = reinterpret_cast<vec2_t<TF>*>(smem_raw);
    if (ld_flag(&ctl->phase_done)) {
        end_loop(h);
        return;
    }
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
    reduce_theta_F(th, fsum, partials, ctl, hist, V, h);
    if (FFT) {
        __syncthreads();
        tile_x_lines<TF, false, LMAX>(d, sm);
        __syncthreads();
        plane_y_lines<TF, false, LMAX>(d, sm, fs, rsx, Fd + s0, V, Lx);
    }
}

// Whether every stored link is within 1e-3 of SU(3) (rows 0,1 orthonormal): the
// range the fixed-point products are bounded for.  A stored row 2 (18-real form) has to be
// the product of rows 0,1 to rounding as well (2^-50; its own error in FP64 is below
// 2^-51): the loop keeps rows 0,1 only.  *wide is set by any other link.
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
    bool ok = fabsf(n0 - 1.f) < 1e-3f && fabsf(n1 - 1.f) < 1e-3f && norm2(ip) < 1e-6f;
    if (d.ne == 9 && ok) {
        bool bad = false;
        cdig rd[6];
#pragma unroll
        for (int e = 0; e < 6; e++) rd[e] = digits(cfx{d2fx<kFxBits>(u[e].re, &bad), d2fx<kFxBits>(u[e].im, &bad)});
#pragma unroll
        for (int j = 0; j < 3; j++) {
            ok = ok && fabs(u[6 + j].re) < 2.0 && fabs(u[6 + j].im) < 2.0;  // false for NaN
            const cfx t = cfx{d2fx<kFxBits>(u[6 + j].re, &bad), d2fx<kFxBits>(u[6 + j].im, &bad)};
            const cfx e = t - fx_row2<3>(rd, rd + 3, j);
            ok = ok && llabs(e.re) <= 1ll << (kFxBits - 50) && llabs(e.im) <= 1ll << (kFxBits - 50);
        }
    }
    if (!ok) *wide = 1;
}

}  // namespace lgf
