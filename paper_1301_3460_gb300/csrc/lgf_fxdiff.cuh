// The derivative of one step on 64-bit fixed point: the products of k_bwd_update
// (lgf_diff.cuh, conventions and formulas there) with links and g from the integer
// forward pass.  The cotangent of a link is scaled by the power of two that puts its
// largest component just below 2^57 (with the pull-back of its third row the rows then
// have norms below 2^61, and the sums of products stay within 64 bits); the products
// are linear in it, so the scale comes off at the end.
#pragma once
#include "lgf_diff.cuh"
#include "lgf_fxt.cuh"

namespace lgf {

// conj(a b)
__device__ __forceinline__ cfx fx_conj_mul(cdig3 a, cdig3 b)
{
    // a x 2^k, b x 2^61: result x 2^k
    const fx p = fval<3>(fmul<3>(a.re, b.re)), q = fval<3>(fmul<3>(a.im, b.im)), r = fval<3>(fmul<3>(a.s, b.s));
    return cfx{p - q, p + q - r};
}

// G_r0, G_r1 += pull-back of G_r2 through r2 = conj(r0 x r1) (row2_bwd)
__device__ __forceinline__ void fx_row2_bwd(const cdig3* r0, const cdig3* r1, const cdig3* g2, cfx* G0, cfx* G1)
{
#pragma unroll
    for (int j = 0; j < 3; j++) {
        const int a = j == 0 ? 1 : j == 1 ? 2 : 0, b = j == 0 ? 2 : j == 1 ? 0 : 1;
        // r2_j = conj(r0_a r1_b - r0_b r1_a)
        G0[a] = G0[a] + fx_conj_mul(g2[j], r1[b]);
        G1[b] = G1[b] + fx_conj_mul(g2[j], r0[a]);
        G0[b] = G0[b] - fx_conj_mul(g2[j], r1[a]);
        G1[a] = G1[a] - fx_conj_mul(g2[j], r0[b]);
    }
}

// conj(a0) b0 + conj(a1) b1 (a with differences, b with sums), x 2^S scale of fval
template <int S> __device__ __forceinline__ cfx fx_dag2(cdig3 a0, cdig3 b0, cdig3 a1, cdig3 b1)
{
    facc p = fmul<S>(a0.re, b0.re), q = fmul<S>(a0.im, b0.im), r = fmul<S>(a0.s, b0.s);
    fmac(p, a1.re, b1.re);
    fmac(q, a1.im, b1.im);
    fmac(r, a1.s, b1.s);
    const fx pv = fval<S>(p), qv = fval<S>(q), rv = fval<S>(r);
    return cfx{pv + qv, rv - pv + qv};  // conj(a) b = (p + q, r - p + q), r = (Re a - Im a)(Re b + Im b)
}

// b1 of lgf_diff.cuh, one thread per link (mu = blockIdx.y).  gX: g x 2^62 of the forward
// pass.  Gp, Gud: [4][9][V].  On entry Gp holds the cotangent of the new links and the first
// six slots of a link in Gud the link itself, x 2^61; on exit Gud holds the direct cotangent
// of U and the first six slots of Gp the link's parts of G_g(x) (rows 0,1).  Q: the
// link's parts of G_g(x+mu).  In FP64 (Gud and Gp are read and written by the link's own
// thread only, and read as what they hold).  The nine components of a cotangent share one scale:
// their errors are 2^-57 of the largest of them, where FP64's are 2^-53 of the largest
// term of each sum.  32^4: 4.00 ms in FP64 (2000 operations per site at 2 per clock and
// SM), 1.50 ms like this (5000 integer products per site; 12 warps per SM at 168
// registers, 16 at 128 take 1.7 ms).
template <int NT, int MB>
__global__ void __launch_bounds__(NT, MB) k_bwd_update_fx(Lat d, const longlong2* __restrict__ g, double2* Gp, double2* Gud,
                                                          double2* __restrict__ Q)
{
    const int V = d.V, mu = blockIdx.y;
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= V) return;
    int c[4];
    site_coords(d, s, c);
    const int sn = site_shift(d, s, mu == 0 ? c[0] : mu == 1 ? c[1] : mu == 2 ? c[2] : c[3], mu, +1);
    // the cotangent and its scale
    double2 gp[9];
    unsigned top = 0;
#pragma unroll
    for (int e = 0; e < 9; e++) {
        gp[e] = Gp[(size_t)(mu * 9 + e) * V + s];
        top = max(top, max((unsigned)__double2hiint(gp[e].x) & 0x7fffffffu, (unsigned)__double2hiint(gp[e].y) & 0x7fffffffu));
    }
    const int ex = (int)(top >> 20) - 1022 + 3;  // components below 2^57
    const bool bad = top >= 0x7ff00000u;
    cfx G[6];
    cdig3 g2[3];
#pragma unroll
    for (int e = 0; e < 6; e++) G[e] = cfx{d2fx_rel(gp[e].x, ex), d2fx_rel(gp[e].y, ex)};
#pragma unroll
    for (int e = 0; e < 3; e++) g2[e] = with_sum(cfx{d2fx_rel(gp[6 + e].x, ex), d2fx_rel(gp[6 + e].y, ex)});
    const double nan = __hiloint2double(0x7ff80000, 0);
    auto put = [&](double2* p, cfx v) {
        *p = bad ? make_double2(nan, nan) : make_double2(fx2d_safe(v.re, 60 - ex), fx2d_safe(v.im, 60 - ex));
    };
    // an entry of the link
    auto link = [&](int e) {
        const double2 v = Gud[(size_t)(mu * 9 + e) * V + s];
        return cfx{__double_as_longlong(v.x), __double_as_longlong(v.y)};
    };
    cdig3 gx[6], Vr[6];  // Vr = rows 0,1 of g(x) U (x 2^61)
#pragma unroll
    for (int e = 0; e < 6; e++) gx[e] = with_sum(ldx(g + (size_t)e * V + s));
    {
        cdig3 ud[9];
#pragma unroll
        for (int e = 0; e < 6; e++) ud[e] = with_sum(link(e));
#pragma unroll
        for (int j = 0; j < 3; j++) ud[6 + j] = with_sum(fx_row2<3>(ud, ud + 3, j));
        cfx t[6];
#pragma unroll
        for (int j = 0; j < 3; j++) {
            t[j] = fx_mul<2>(gx, ud, j);
            t[3 + j] = fx_mul<2>(gx + 3, ud, j);
        }
        // Up = Vr gn^dag, rows 0,1 (x 2^61), and the pull-back of the cotangent's row 2
        cdig3 vd[6], up[6];
#pragma unroll
        for (int e = 0; e < 6; e++) {
            Vr[e] = with_sum(t[e]);
            vd[e] = cdig3{Vr[e].re, Vr[e].im, digits(t[e].re - t[e].im)};
        }
#pragma unroll
        for (int j = 0; j < 3; j++) {
            cdig3 b[3];
#pragma unroll
            for (int k = 0; k < 3; k++) b[k] = with_sum(ldx(g + (size_t)(3 * j + k) * V + sn));
            up[j] = with_sum(fx_mul_dag<2>(vd, b));
            up[3 + j] = with_sum(fx_mul_dag<2>(vd + 3, b));
        }
        fx_row2_bwd(up, up + 3, g2, G, G + 3);
    }
    // Y = G01 gn
    cfx Y[6];
    {
        cdig3 Gs[6];
#pragma unroll
        for (int e = 0; e < 6; e++) Gs[e] = with_sum(G[e]);
        cdig3 b[9];
#pragma unroll
        for (int e = 0; e < 9; e++) b[e] = with_sum(ldx(g + (size_t)e * V + sn));
#pragma unroll
        for (int j = 0; j < 3; j++) {
            Y[j] = fx_mul<2>(Gs, b, j);
            Y[3 + j] = fx_mul<2>(Gs + 3, b, j);
        }
    }
    // Q = G01^dag Vr: the contribution to G_g(x+mu)
    {
        cdig3 Gd[6];
#pragma unroll
        for (int e = 0; e < 6; e++) Gd[e] = with_diff(G[e]);
#pragma unroll
        for (int a = 0; a < 3; a++)
#pragma unroll
            for (int b = 0; b < 3; b++)
                put(Q + (size_t)(mu * 9 + 3 * a + b) * V + s, fx_dag2<3>(Gd[a], Vr[b], Gd[3 + a], Vr[3 + b]));
    }
    // G_g(x) rows 0,1 += Y U^dag
    {
        cdig3 Yd[6], ud[9];
#pragma unroll
        for (int e = 0; e < 6; e++) {
            Yd[e] = with_diff(Y[e]);
            ud[e] = with_sum(link(e));
        }
#pragma unroll
        for (int j = 0; j < 3; j++) ud[6 + j] = with_sum(fx_row2<3>(ud, ud + 3, j));
#pragma unroll
        for (int j = 0; j < 3; j++) {
            put(Gp + (size_t)(mu * 9 + j) * V + s, fx_mul_dag<3>(Yd, ud + 3 * j));
            put(Gp + (size_t)(mu * 9 + 3 + j) * V + s, fx_mul_dag<3>(Yd + 3, ud + 3 * j));
        }
    }
    // G_U^direct = (rows 0,1 of g)^dag Y
    {
        cdig3 Ys[6];
#pragma unroll
        for (int e = 0; e < 6; e++) Ys[e] = with_sum(Y[e]);
#pragma unroll
        for (int a = 0; a < 3; a++) {
            const cdig3 a0 = cdig3{gx[a].re, gx[a].im, digits(value(gx[a].re) - value(gx[a].im))};
            const cdig3 a1 = cdig3{gx[3 + a].re, gx[3 + a].im, digits(value(gx[3 + a].re) - value(gx[3 + a].im))};
#pragma unroll
            for (int b = 0; b < 3; b++)
                put(Gud + (size_t)(mu * 9 + 3 * a + b) * V + s, fx_dag2<2>(a0, Ys[b], a1, Ys[3 + b]));
        }
    }
}

}  // namespace lgf
