// Wilson-action Monte Carlo of the links a context holds: SU(3) configurations
// of the kind the paper's 32^4 comparison runs gauge-fix (Wilson action at three
// couplings), generated on the device so that they go straight into the fixing
// loop.  The paper does not describe its generator; this one is the standard
// Cabibbo-Marinari heat bath with overrelaxation.
//
// Action S = beta sum_P (1 - Re Tr U_P / 3).  The links U_mu(x) with x of one
// checkerboard parity share no plaquette, so one launch updates all of them at
// once: one thread per site of that parity, direction mu fixed per launch.  Per
// link, with the staple sum
//   A = sum_{nu != mu} U_nu(x+mu) U_mu(x+nu)^dag U_nu(x)^dag
//                    + U_nu(x+mu-nu)^dag U_mu(x-nu)^dag U_nu(x-nu),
// W = U A and the SU(2) subgroups (0,1), (0,2), (1,2) in turn: the 2x2 block w
// of W gives r = (w_ii + conj w_jj)/2, s = (w_ij - conj w_ji)/2, k = |(r, s)|
// and the SU(2) element V = [[r, s], [-conj s, conj r]]/k, and the link becomes
// R U with R in the subgroup:
//   heat bath      R = Y V^dag, Y ~ sqrt(1 - y0^2) exp(b y0), b = 2 beta k / 3,
//                  uniform direction (Kennedy-Pendleton for b >= 1.6, Creutz
//                  below, where their acceptance rates cross)
//   overrelaxation R = (V^dag)^2 (leaves Re Tr(U A) unchanged)
// then rows 0,1 are Gram-Schmidt orthonormalised and row 2 rebuilt.
//
// Random numbers are counter-based (Philox4x32-10, Salmon et al., SC'11): key =
// the 64-bit seed, counter (mu V + s, sweep, 1024 subgroup + draw, 0), so a
// result depends on neither the launch shape nor the thread order.  Attempt a of
// subgroup g reads draw 2a (y0) and, once accepted, 2a + 1 (direction); after
// 512 failed attempts the subgroup is left unchanged.
//
// Per link: 12 3x3 complex products for the staples (the six of two SU(3) links with
// row 2 rebuilt instead of multiplied out), one for W, the rotations and the
// sampler's transcendental functions.  In FP64 (k_wilson) the FP64 pipe bounds it (2
// operations per clock and SM); by default the products, rotations and the
// re-orthonormalisation run on 64-bit fixed point (k_wilson_fx, lgf_fx.cuh: finer
// than FP64 for matrices bounded by 1), with the SU(2) elements and the sampler in
// FP64.  Links outside the fixed-point range take the FP64 kernel.
#include <cuda_runtime.h>
#include <stdint.h>

#include "lgf_common.cuh"
#include "lgf_fx.cuh"
#include "lgf_kernels.cuh"
#include "lgf_launch.h"

namespace lgf {
namespace {

using C = cx<double>;

constexpr int kWilsonThreads = 128;
constexpr int kPlaqThreads = 256;
constexpr int kPlaqBlocks = 1216;  // 8 per SM on 152 SMs; grid-stride beyond

// matrix helpers for T = double (the FP64 generator) and T = float (the staples
// of the FP32 one); links are FP64 in memory in both cases

template <typename T> __device__ __forceinline__ cx<T> ldl(const double2* p)
{
    const double2 v = __ldg(p);
    return mk<T>((T)v.x, (T)v.y);
}
template <typename T> __device__ __forceinline__ cx<T> ldl(const float2* p)
{
    const float2 v = __ldg(p);
    return mk<T>((T)v.x, (T)v.y);
}

template <typename T, typename S>
__device__ __forceinline__ void load3(const S* __restrict__ U, int V, int ne, int mu, int s, cx<T>* m)
{
#pragma unroll
    for (int e = 0; e < 6; e++) m[e] = ldl<T>(U + (size_t)(mu * ne + e) * V + s);
    if (ne == 9) {
#pragma unroll
        for (int e = 6; e < 9; e++) m[e] = ldl<T>(U + (size_t)(mu * 9 + e) * V + s);
    } else {
        complete_row2(m, m + 6);
    }
}

// rows 0,1 of a link (all that a product whose row 2 is rebuilt needs)
template <typename T, typename S>
__device__ __forceinline__ void load2(const S* __restrict__ U, int V, int ne, int mu, int s, cx<T>* m)
{
#pragma unroll
    for (int e = 0; e < 6; e++) m[e] = ldl<T>(U + (size_t)(mu * ne + e) * V + s);
}

// c = a b for a, b in SU(3): rows 0,1 multiplied out, row 2 = conj(row0 x row1)
// (a's row 2 is not read)
template <typename T> __device__ __forceinline__ void mm_su3(const cx<T>* a, const cx<T>* b, cx<T>* c)
{
#pragma unroll
    for (int i = 0; i < 2; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) {
            cx<T> t = cmul(a[3 * i], b[j]);
            t = cmac(t, a[3 * i + 1], b[3 + j]);
            c[3 * i + j] = cmac(t, a[3 * i + 2], b[6 + j]);
        }
    complete_row2(c, c + 6);
}

// c = a b
template <typename T> __device__ __forceinline__ void mm(const cx<T>* a, const cx<T>* b, cx<T>* c)
{
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) {
            cx<T> t = cmul(a[3 * i], b[j]);
            t = cmac(t, a[3 * i + 1], b[3 + j]);
            c[3 * i + j] = cmac(t, a[3 * i + 2], b[6 + j]);
        }
}

// acc += a b^dag
template <typename T> __device__ __forceinline__ void mm_nd_acc(const cx<T>* a, const cx<T>* b, cx<T>* acc)
{
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) {
            cx<T> t = acc[3 * i + j];
#pragma unroll
            for (int k = 0; k < 3; k++) t = cmacc(t, a[3 * i + k], b[3 * j + k]);
            acc[3 * i + j] = t;
        }
}

// acc += a^dag b
template <typename T> __device__ __forceinline__ void mm_dn_acc(const cx<T>* a, const cx<T>* b, cx<T>* acc)
{
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) {
            cx<T> t = acc[3 * i + j];
#pragma unroll
            for (int k = 0; k < 3; k++) t = cmacc(t, b[3 * k + j], a[3 * k + i]);
            acc[3 * i + j] = t;
        }
}

// staple sum A of link (mu, s) of parity c
template <typename T, typename S>
__device__ __forceinline__ void staple_sum(const Lat& d, const S* __restrict__ U, int mu, int s, const int* c,
                                           cx<T>* A)
{
    const int V = d.V, ne = d.ne;
#pragma unroll
    for (int e = 0; e < 9; e++) A[e] = mk<T>(0, 0);
    const int sp = site_shift(d, s, c[mu], mu, +1);
#pragma unroll
    for (int nu = 0; nu < 4; nu++) {
        if (nu == mu) continue;
        const int snp = site_shift(d, s, c[nu], nu, +1);
        const int snm = site_shift(d, s, c[nu], nu, -1);
        const int spm = site_shift(d, sp, c[nu], nu, -1);  // x + mu - nu
        cx<T> a[9], b[9], q[9];
        load2<T>(U, V, ne, nu, s, a);
        load3<T>(U, V, ne, mu, snp, b);
        mm_su3<T>(a, b, q);             // U_nu(x) U_mu(x+nu)
        load3<T>(U, V, ne, nu, sp, a);
        mm_nd_acc<T>(a, q, A);          // + U_nu(x+mu) q^dag
        load2<T>(U, V, ne, mu, snm, a);
        load3<T>(U, V, ne, nu, spm, b);
        mm_su3<T>(a, b, q);             // U_mu(x-nu) U_nu(x+mu-nu)
        load3<T>(U, V, ne, nu, snm, a);
        mm_dn_acc<T>(q, a, A);          // + q^dag U_nu(x-nu)
    }
}

// ---------------------------------------------------------------- Philox4x32-10

__device__ __forceinline__ void philox(uint32_t c[4], uint32_t k0, uint32_t k1)
{
#pragma unroll
    for (int r = 0; r < 10; r++) {
        const uint32_t lo0 = 0xD2511F53u * c[0], hi0 = __umulhi(0xD2511F53u, c[0]);
        const uint32_t lo1 = 0xCD9E8D57u * c[2], hi1 = __umulhi(0xCD9E8D57u, c[2]);
        const uint32_t n0 = hi1 ^ c[1] ^ k0, n2 = hi0 ^ c[3] ^ k1;
        c[0] = n0;
        c[1] = lo1;
        c[2] = n2;
        c[3] = lo0;
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
}

// four uniforms (word + 1/2) 2^-32 in (0, 1), exact in FP64
__device__ __forceinline__ void draw4(uint32_t k0, uint32_t k1, uint32_t link, uint32_t sweep, uint32_t n, double u[4])
{
    uint32_t c[4] = {link, sweep, n, 0u};
    philox(c, k0, k1);
#pragma unroll
    for (int i = 0; i < 4; i++) u[i] = fma((double)c[i], 0x1p-32, 0x1p-33);
}

// y = (y0, y1, y2, y3) with y0 ~ sqrt(1 - y0^2) exp(b y0) on [-1, 1] and the
// direction uniform on the 2-sphere; the identity after 512 failed attempts.
__device__ __noinline__ void su2_draw(double b, uint32_t k0, uint32_t k1, uint32_t link, uint32_t sweep, int sub,
                                      double y[4])
{
    const bool kp = b >= 1.6;
    const double ib = b > 0 ? 1.0 / b : 0.0;
    const double e2b = kp ? 0.0 : expm1(-2.0 * b);
    for (int a = 0; a < 512; a++) {
        double u[4];
        draw4(k0, k1, link, sweep, (uint32_t)(1024 * sub + 2 * a), u);
        double y0;
        bool ok;
        if (kp) {
            // Kennedy-Pendleton: lambda^2 = (an Exp(1) + half a squared normal) / 2b
            const double c = cospi(2.0 * u[1]);
            const double lam2 = -(log(u[0]) + c * c * log(u[2])) * (0.5 * ib);
            ok = u[3] * u[3] <= 1.0 - lam2;
            y0 = 1.0 - 2.0 * lam2;
        } else {
            // Creutz: proposal exp(b y0) by its inverse distribution function
            y0 = b > 0 ? 1.0 + log1p((1.0 - u[0]) * e2b) * ib : 2.0 * u[0] - 1.0;
            ok = u[1] * u[1] <= 1.0 - y0 * y0;
        }
        if (ok) {
            double v[4];
            draw4(k0, k1, link, sweep, (uint32_t)(1024 * sub + 2 * a + 1), v);
            const double ct = 2.0 * v[0] - 1.0;
            const double st = sqrt(1.0 - ct * ct);
            double sp, cp;
            sincospi(2.0 * v[1], &sp, &cp);
            const double rr = sqrt(fmax(1.0 - y0 * y0, 0.0));
            y[0] = y0;
            y[1] = rr * st * cp;
            y[2] = rr * st * sp;
            y[3] = rr * ct;
            return;
        }
    }
    y[0] = 1.0;
    y[1] = y[2] = y[3] = 0.0;
}

// rows i, j of m <- R (rows i, j)
template <int I, int J, typename T>
__device__ __forceinline__ void rot_rows(cx<T>* m, cx<T> R00, cx<T> R01, cx<T> R10, cx<T> R11)
{
#pragma unroll
    for (int c = 0; c < 3; c++) {
        const cx<T> mi = m[3 * I + c], mj = m[3 * J + c];
        m[3 * I + c] = cmac(cmul(R00, mi), R01, mj);
        m[3 * J + c] = cmac(cmul(R10, mi), R11, mj);
    }
}

template <int MODE, int I, int J>
__device__ __forceinline__ void subgroup(C* u, C* w, double beta23, uint32_t k0, uint32_t k1, uint32_t link,
                                         uint32_t sweep, int sub)
{
    const C wii = w[3 * I + I], wjj = w[3 * J + J], wij = w[3 * I + J], wji = w[3 * J + I];
    const C r = mk(0.5 * (wii.re + wjj.re), 0.5 * (wii.im - wjj.im));
    const C s = mk(0.5 * (wij.re - wji.re), 0.5 * (wij.im + wji.im));
    const double k2 = r.re * r.re + r.im * r.im + s.re * s.re + s.im * s.im;
    if (!(k2 > 0)) return;
    const double ik = rsqrt(k2);
    const C a = r * ik, b = s * ik;
    C R00, R01, R10, R11;
    if (MODE == 0) {
        double y[4];
        su2_draw(beta23 * (k2 * ik), k0, k1, link, sweep, sub, y);
        // Y = y0 + i (y1 s1 + y2 s2 + y3 s3); R = Y V^dag, V^dag = [[conj a, -b], [conj b, a]]
        const C Y00 = mk(y[0], y[3]), Y01 = mk(y[2], y[1]), Y10 = mk(-y[2], y[1]), Y11 = mk(y[0], -y[3]);
        const C nb = mk(-b.re, -b.im);
        R00 = cmac(cmul(Y00, conjg(a)), Y01, conjg(b));
        R01 = cmac(cmul(Y00, nb), Y01, a);
        R10 = cmac(cmul(Y10, conjg(a)), Y11, conjg(b));
        R11 = cmac(cmul(Y10, nb), Y11, a);
    } else {
        // R = (V^dag)^2
        const C D00 = conjg(a), D01 = mk(-b.re, -b.im), D10 = conjg(b), D11 = a;
        R00 = cmac(cmul(D00, D00), D01, D10);
        R01 = cmac(cmul(D00, D01), D01, D11);
        R10 = cmac(cmul(D10, D00), D11, D10);
        R11 = cmac(cmul(D10, D01), D11, D11);
    }
    rot_rows<I, J>(u, R00, R01, R10, R11);
    rot_rows<I, J>(w, R00, R01, R10, R11);
}

// Gram-Schmidt of rows 0, 1 (row 2 untouched)
__device__ __forceinline__ void orthonormal_rows01(C* m)
{
    double n0 = 0;
#pragma unroll
    for (int c = 0; c < 3; c++) n0 += norm2(m[c]);
    n0 = rsqrt(n0);
#pragma unroll
    for (int c = 0; c < 3; c++) m[c] = m[c] * n0;
    C ip = mk(0.0, 0.0);
#pragma unroll
    for (int c = 0; c < 3; c++) ip = cmacc(ip, m[3 + c], m[c]);  // sum conj(row0) row1
    double n1 = 0;
#pragma unroll
    for (int c = 0; c < 3; c++) {
        m[3 + c] = m[3 + c] - cmul(ip, m[c]);
        n1 += norm2(m[3 + c]);
    }
    n1 = rsqrt(n1);
#pragma unroll
    for (int c = 0; c < 3; c++) m[3 + c] = m[3 + c] * n1;
}

// Gram-Schmidt of rows 0, 1 and row 2 = conj(row0 x row1)
__device__ __forceinline__ void reunit(C* m)
{
    orthonormal_rows01(m);
    complete_row2(m, m + 6);
}

template <int MODE>
__global__ void __launch_bounds__(kWilsonThreads) k_wilson(Lat d, double2* __restrict__ U, int mu, int parity,
                                                           double beta, uint32_t k0, uint32_t k1, uint32_t sweep)
{
    const int h = blockIdx.x * blockDim.x + threadIdx.x;
    if (h >= (d.V >> 1)) return;
    // site of the given parity with pair index h = s / 2 (Lx is even)
    const int hx = d.L[0] >> 1;
    int c[4];
    int r = h / hx;
    const int xh = h - r * hx;
    c[1] = r % d.L[1];
    r /= d.L[1];
    c[2] = r % d.L[2];
    c[3] = r / d.L[2];
    c[0] = 2 * xh + ((parity + c[1] + c[2] + c[3]) & 1);
    const int s = c[0] + d.stride[1] * c[1] + d.stride[2] * c[2] + d.stride[3] * c[3];
    const int V = d.V, ne = d.ne;

    C A[9];
    staple_sum<double>(d, U, mu, s, c, A);
    C u[9], w[9];
    load3<double>(U, V, ne, mu, s, u);
    mm<double>(u, A, w);
    const uint32_t link = (uint32_t)mu * (uint32_t)V + (uint32_t)s;
    const double beta23 = beta * (2.0 / 3.0);  // b = 2 beta k / 3
    subgroup<MODE, 0, 1>(u, w, beta23, k0, k1, link, sweep, 0);
    subgroup<MODE, 0, 2>(u, w, beta23, k0, k1, link, sweep, 1);
    subgroup<MODE, 1, 2>(u, w, beta23, k0, k1, link, sweep, 2);
    reunit(u);
#pragma unroll
    for (int e = 0; e < 6; e++) st<double>(U + (size_t)(mu * ne + e) * V + s, u[e]);
    if (ne == 9) {
#pragma unroll
        for (int e = 6; e < 9; e++) st<double>(U + (size_t)(mu * 9 + e) * V + s, u[e]);
    }
}

// ---------------------------------------------------------------- fixed-point generator

// The links of a call on the grid 2^-61, all three rows: [mu][9][V] (the rows saved
// from rebuilding, 144 integer products per staple, cost half as many bytes again).
// Staples of up to six unit matrices and W are kept x 2^58 (range +-32).
// They begin where the FP64 links do and reach into the idle arrays behind them: a thread
// converts the four links of its site, the last direction first on the way in (nothing is
// overwritten before it is read) and the first one first on the way back.

__global__ void k_links_to_fx(Lat d, const longlong2* U, longlong2* UX)
{
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= d.V) return;
#pragma unroll 1
    for (int mu = 3; mu >= 0; mu--) {
        cfx r[6];
        cdig rd[6];
#pragma unroll
        for (int e = 0; e < 6; e++) {
            const longlong2 v = U[(size_t)(mu * d.ne + e) * d.V + s];
            r[e] = cfx{d2fx_rn<kFxBits>(__longlong_as_double(v.x)), d2fx_rn<kFxBits>(__longlong_as_double(v.y))};
            rd[e] = digits(r[e]);
        }
#pragma unroll
        for (int e = 0; e < 6; e++) stx(UX + (size_t)(mu * 9 + e) * d.V + s, r[e]);
#pragma unroll
        for (int j = 0; j < 3; j++) stx(UX + (size_t)(mu * 9 + 6 + j) * d.V + s, fx_row2<3>(rd, rd + 3, j));
    }
}
__global__ void k_links_from_fx(Lat d, const longlong2* UX, double2* U)
{
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= d.V) return;
#pragma unroll 1
    for (int mu = 0; mu < 4; mu++) {
        cx<double> w[9];
#pragma unroll
        for (int e = 0; e < 6; e++) {
            const cfx v = ldv<fx>(UX + (size_t)(mu * 9 + e) * d.V + s);
            w[e] = mk<double>(fx2d(v.re, kFxBits), fx2d(v.im, kFxBits));
        }
        if (d.ne == 9) complete_row2(w, w + 6);
        // the loads come first whatever types the two views of the place have
        asm volatile("" ::: "memory");
        store_link<double>(U, d.V, d.ne, mu, s, w);
        asm volatile("" ::: "memory");
    }
}

__device__ __forceinline__ void load9x(const longlong2* __restrict__ U, int V, int mu, int s, cfx* m)
{
#pragma unroll
    for (int e = 0; e < 9; e++) m[e] = ldv<fx>(U + (size_t)(mu * 9 + e) * V + s);
}

// q = a b for SU(3) links a (rows 0,1 read), b; row 2 rebuilt
__device__ __forceinline__ void fx_mm_su3(const longlong2* __restrict__ U, int V, int mua, int sa, int mub, int sb, cfx* q)
{
    cdig3 a[6], b[9];
#pragma unroll
    for (int e = 0; e < 6; e++) a[e] = with_sum(ldv<fx>(U + (size_t)(mua * 9 + e) * V + sa));
#pragma unroll
    for (int e = 0; e < 9; e++) b[e] = with_sum(ldv<fx>(U + (size_t)(mub * 9 + e) * V + sb));
#pragma unroll
    for (int j = 0; j < 3; j++) {
        q[j] = fx_mul<3>(a, b, j);
        q[3 + j] = fx_mul<3>(a + 3, b, j);
    }
    cdig qd[6];
#pragma unroll
    for (int e = 0; e < 6; e++) qd[e] = digits(q[e]);
#pragma unroll
    for (int j = 0; j < 3; j++) q[6 + j] = fx_row2<3>(qd, qd + 3, j);
}

// staple sum of link (mu, s), x 2^58
__device__ __forceinline__ void fx_staple_sum(const Lat& d, const longlong2* __restrict__ U, int mu, int s, const int* c,
                                              cfx* A)
{
    const int V = d.V;
#pragma unroll
    for (int e = 0; e < 9; e++) A[e] = cfx{0, 0};
    const int sp = site_shift(d, s, c[mu], mu, +1);
#pragma unroll 1
    for (int nu = 0; nu < 4; nu++) {
        if (nu == mu) continue;
        const int cn = nu == 0 ? c[0] : nu == 1 ? c[1] : nu == 2 ? c[2] : c[3];
        // x + mu has the same nu coordinate as x
        const int up = site_shift(d, s, cn, nu, +1), dn = site_shift(d, s, cn, nu, -1);
        const int dnp = site_shift(d, sp, cn, nu, -1);
        cfx q[9];
        fx_mm_su3(U, V, nu, s, mu, up, q);  // U_nu(x) U_mu(x+nu)
        {
            // + U_nu(x+mu) q^dag
            cdig3 qd[9];
#pragma unroll
            for (int e = 0; e < 9; e++) qd[e] = with_sum(q[e]);
#pragma unroll
            for (int i = 0; i < 3; i++) {
                cdig3 a[3];
#pragma unroll
                for (int k = 0; k < 3; k++) a[k] = with_diff(ldv<fx>(U + (size_t)(nu * 9 + 3 * i + k) * V + sp));
#pragma unroll
                for (int j = 0; j < 3; j++) A[3 * i + j] = A[3 * i + j] + fx_mul_dag<0>(a, qd + 3 * j);
            }
        }
        fx_mm_su3(U, V, mu, dn, nu, dnp, q);  // U_mu(x-nu) U_nu(x+mu-nu)
        {
            // + q^dag U_nu(x-nu): conj(q_ki) b_kj = conj(q_ki conj(b_kj))
            cdig3 qd[9];
#pragma unroll
            for (int e = 0; e < 9; e++) qd[e] = with_diff(q[e]);
#pragma unroll
            for (int j = 0; j < 3; j++) {
                cdig3 b[3];
#pragma unroll
                for (int k = 0; k < 3; k++) b[k] = with_sum(ldv<fx>(U + (size_t)(nu * 9 + 3 * k + j) * V + dn));
#pragma unroll
                for (int i = 0; i < 3; i++) {
                    const cdig3 a[3] = {qd[i], qd[3 + i], qd[6 + i]};
                    const cfx t = fx_mul_dag<0>(a, b);
                    A[3 * i + j] = A[3 * i + j] + cfx{t.re, -t.im};
                }
            }
        }
    }
}

// R = [[a, b], [-conj b, conj a]], x 2^61: a with its sum and difference, b likewise
struct fx_su2 {
    cdig3 as, ad, bs, bd;
};
// R00 x + R01 y (x, y with sums)
template <int S> __device__ __forceinline__ cfx fx_rot0(const fx_su2& R, cdig3 x, cdig3 y)
{
    facc p = fmul<S>(R.as.re, x.re), q = fmul<S>(R.as.im, x.im), r = fmul<S>(R.as.s, x.s);
    fmac(p, R.bs.re, y.re);
    fmac(q, R.bs.im, y.im);
    fmac(r, R.bs.s, y.s);
    const fx pv = fval<S>(p), qv = fval<S>(q), rv = fval<S>(r);
    return cfx{pv - qv, rv - pv - qv};
}
// R10 x + R11 y = conj(a) y - conj(b) x, with conj(u) v = (p + q, r - p + q), r = (Re u - Im u)(Re v + Im v)
template <int S> __device__ __forceinline__ cfx fx_rot1(const fx_su2& R, cdig3 x, cdig3 y)
{
    facc p = fmul<S>(R.ad.re, y.re), q = fmul<S>(R.ad.im, y.im), r = fmul<S>(R.ad.s, y.s);
    facc p2 = fmul<S>(R.bd.re, x.re), q2 = fmul<S>(R.bd.im, x.im), r2 = fmul<S>(R.bd.s, x.s);
    const fx pv = fval<S>(p) - fval<S>(p2), qv = fval<S>(q) - fval<S>(q2), rv = fval<S>(r) - fval<S>(r2);
    return cfx{pv + qv, rv - pv + qv};
}

// the SU(2) rotation of the block (wii, wij; wji, wjj) of W (x 2^58): R = Y V^dag (heat
// bath) or (V^dag)^2; false where the block projects to zero
template <int MODE>
__device__ __forceinline__ bool fx_subgroup(cfx wii, cfx wij, cfx wji, cfx wjj, double beta23, uint32_t k0, uint32_t k1,
                                            uint32_t link, uint32_t sweep, int sub, fx_su2& R)
{
    // r = (wii + conj wjj)/2, s = (wij - conj wji)/2: sums exact, x 2^59
    const double rr = fx2d(wii.re + wjj.re, kFxSum + 1), ri = fx2d(wii.im - wjj.im, kFxSum + 1);
    const double sr = fx2d(wij.re - wji.re, kFxSum + 1), si = fx2d(wij.im + wji.im, kFxSum + 1);
    const double k2 = rr * rr + ri * ri + sr * sr + si * si;
    if (!(k2 > 0)) return false;
    const double ik = rsqrt(k2);
    const C a = mk(rr * ik, ri * ik), b = mk(sr * ik, si * ik);  // V = [[a, b], [-conj b, conj a]]
    C R00, R01;
    if (MODE == 0) {
        double y[4];
        su2_draw(beta23 * (k2 * ik), k0, k1, link, sweep, sub, y);
        // Y = y0 + i (y1 s1 + y2 s2 + y3 s3); V^dag = [[conj a, -b], [conj b, a]]
        const C Y00 = mk(y[0], y[3]), Y01 = mk(y[2], y[1]);
        R00 = cmac(cmul(Y00, conjg(a)), Y01, conjg(b));
        R01 = cmac(cmul(Y00, mk(-b.re, -b.im)), Y01, a);
    } else {
        // (V^dag)^2: conj(a)^2 - |b|^2, -b (a + conj a)
        R00 = mk(fma(a.re, a.re, -fma(a.im, a.im, norm2(b))), -2.0 * a.re * a.im);
        R01 = b * (-2.0 * a.re);
    }
    bool bad = false;
    const cfx x = cfx{d2fx<kFxBits>(R00.re, &bad), d2fx<kFxBits>(R00.im, &bad)};
    const cfx y = cfx{d2fx<kFxBits>(R01.re, &bad), d2fx<kFxBits>(R01.im, &bad)};
    R.as = with_sum(x);
    R.ad = with_diff(x);
    R.bs = with_sum(y);
    R.bd = with_diff(y);
    return true;
}

// Of W only what the later subgroups read is rotated (seven entries), of the link
// rows 0,1 and, for the second subgroup, row 2.  Sweeps at 32^4: overrelaxation 14.4 ms
// in FP64, 3.8 ms like this (integer products); heat bath 19.6 and 8.8 ms (what it
// takes beyond the overrelaxation is the sampler).  Attempts are not what costs there:
// passing over those that FP32 rules out, and one direction per warp after the loop,
// left the sweep at 8.3 ms under the profiler, as without.
template <int MODE>
__global__ void __launch_bounds__(kWilsonThreads, 3) k_wilson_fx(Lat d, longlong2* __restrict__ U, int mu, int parity,
                                                              double beta, uint32_t k0, uint32_t k1, uint32_t sweep)
{
    const int h = blockIdx.x * blockDim.x + threadIdx.x;
    if (h >= (d.V >> 1)) return;
    const int hx = d.L[0] >> 1;
    int c[4];
    int r = h / hx;
    const int xh = h - r * hx;
    c[1] = r % d.L[1];
    r /= d.L[1];
    c[2] = r % d.L[2];
    c[3] = r / d.L[2];
    c[0] = 2 * xh + ((parity + c[1] + c[2] + c[3]) & 1);
    const int s = c[0] + d.stride[1] * c[1] + d.stride[2] * c[2] + d.stride[3] * c[3];
    const int V = d.V;
    cfx A[9], u[9], w[9];
    fx_staple_sum(d, U, mu, s, c, A);
    load9x(U, V, mu, s, u);
    {
        cdig3 Ad[9];
#pragma unroll
        for (int e = 0; e < 9; e++) Ad[e] = with_sum(A[e]);
#pragma unroll
        for (int i = 0; i < 3; i++) {
            const cdig3 ud[3] = {with_sum(u[3 * i]), with_sum(u[3 * i + 1]), with_sum(u[3 * i + 2])};
#pragma unroll
            for (int j = 0; j < 3; j++) w[3 * i + j] = fx_mul<3>(ud, Ad, j);
        }
    }
    const uint32_t link = (uint32_t)mu * (uint32_t)V + (uint32_t)s;
    const double beta23 = beta * (2.0 / 3.0);
    fx_su2 R;
    if (fx_subgroup<MODE>(w[0], w[1], w[3], w[4], beta23, k0, k1, link, sweep, 0, R)) {
#pragma unroll
        for (int j = 0; j < 3; j++) {
            const cdig3 x = with_sum(w[j]), y = with_sum(w[3 + j]);
            const cfx n = fx_rot0<3>(R, x, y);
            if (j > 0) w[3 + j] = fx_rot1<3>(R, x, y);
            w[j] = n;
        }
#pragma unroll
        for (int j = 0; j < 3; j++) {
            const cdig3 x = with_sum(u[j]), y = with_sum(u[3 + j]);
            u[j] = fx_rot0<3>(R, x, y);
            u[3 + j] = fx_rot1<3>(R, x, y);
        }
    }
    if (fx_subgroup<MODE>(w[0], w[2], w[6], w[8], beta23, k0, k1, link, sweep, 1, R)) {
#pragma unroll
        for (int j = 1; j < 3; j++) w[6 + j] = fx_rot1<3>(R, with_sum(w[j]), with_sum(w[6 + j]));
#pragma unroll
        for (int j = 0; j < 3; j++) {
            const cdig3 x = with_sum(u[j]), y = with_sum(u[6 + j]);
            u[j] = fx_rot0<3>(R, x, y);
            u[6 + j] = fx_rot1<3>(R, x, y);
        }
    }
    if (fx_subgroup<MODE>(w[4], w[5], w[7], w[8], beta23, k0, k1, link, sweep, 2, R)) {
#pragma unroll
        for (int j = 0; j < 3; j++) u[3 + j] = fx_rot0<3>(R, with_sum(u[3 + j]), with_sum(u[6 + j]));
    }
    // rows 0,1 orthonormalised, rounded to the nearest double (exact in FP64, so that a
    // chain does not depend on how it is split into calls), row 2 rebuilt.  Measured rms of
    // <row 0, row 1>: 3.3e-17 for rough links, 1.4e-17 near 1; with every entry on the grid
    // 2^-53 both are 6.4e-17.
    cfx X[6], o[6];
    cdig od[6];
#pragma unroll
    for (int e = 0; e < 6; e++) X[e] = cfx{(u[e].re + 1) >> 1, (u[e].im + 1) >> 1};
    fx_gram_schmidt(X, 1, o, od);
#pragma unroll
    for (int e = 0; e < 6; e++) {
        o[e] = cfx{fx_round_double(o[e].re), fx_round_double(o[e].im)};
        od[e] = digits(o[e]);
        stx(U + (size_t)(mu * 9 + e) * V + s, o[e]);
    }
#pragma unroll
    for (int j = 0; j < 3; j++) stx(U + (size_t)(mu * 9 + 6 + j) * V + s, fx_row2<3>(od, od + 3, j));
}

// ---------------------------------------------------------------- FP32 generator

// The same update with the staples, W, the SU(2) draws and the rotation of the
// link in FP32, all read from the FP32 copy (links stay FP64 in memory: rows 0,1
// of the rotated link are re-orthonormalised in FP64, so the stored link stays in
// SU(3) to FP64 rounding).  A Markov chain of its own:
// the heat bath samples exp((beta/3) Re Tr(U A)) with A known to FP32 rounding,
// and its uniforms take the top 24 bits of the same Philox words.

__device__ __forceinline__ void draw4f(uint32_t k0, uint32_t k1, uint32_t link, uint32_t sweep, uint32_t n, float u[4])
{
    uint32_t c[4] = {link, sweep, n, 0u};
    philox(c, k0, k1);
#pragma unroll
    for (int i = 0; i < 4; i++) u[i] = fmaf((float)(c[i] >> 8), 0x1p-24f, 0x1p-25f);
}

__device__ __noinline__ void su2_draw_f(float b, uint32_t k0, uint32_t k1, uint32_t link, uint32_t sweep, int sub,
                                        float y[4])
{
    const bool kp = b >= 1.6f;
    const float ib = b > 0 ? 1.0f / b : 0.0f;
    const float e2b = kp ? 0.0f : expm1f(-2.0f * b);
    for (int a = 0; a < 512; a++) {
        float u[4];
        draw4f(k0, k1, link, sweep, (uint32_t)(1024 * sub + 2 * a), u);
        float y0;
        bool ok;
        if (kp) {
            const float c = cospif(2.0f * u[1]);
            const float lam2 = -(logf(u[0]) + c * c * logf(u[2])) * (0.5f * ib);
            ok = u[3] * u[3] <= 1.0f - lam2;
            y0 = 1.0f - 2.0f * lam2;
        } else {
            y0 = b > 0 ? 1.0f + log1pf((1.0f - u[0]) * e2b) * ib : 2.0f * u[0] - 1.0f;
            ok = u[1] * u[1] <= 1.0f - y0 * y0;
        }
        if (ok) {
            float v[4];
            draw4f(k0, k1, link, sweep, (uint32_t)(1024 * sub + 2 * a + 1), v);
            const float ct = 2.0f * v[0] - 1.0f;
            const float st = sqrtf(fmaxf(1.0f - ct * ct, 0.0f));
            float sp, cp;
            sincospif(2.0f * v[1], &sp, &cp);
            const float rr = sqrtf(fmaxf(1.0f - y0 * y0, 0.0f));
            y[0] = y0;
            y[1] = rr * st * cp;
            y[2] = rr * st * sp;
            y[3] = rr * ct;
            return;
        }
    }
    y[0] = 1.0f;
    y[1] = y[2] = y[3] = 0.0f;
}

// rows i, j of w and of the link u (both FP32 here) <- R (rows i, j)
template <int MODE, int I, int J>
__device__ __forceinline__ void subgroup32(cx<float>* u, cx<float>* w, float beta23, uint32_t k0, uint32_t k1,
                                           uint32_t link, uint32_t sweep, int sub)
{
    using F = cx<float>;
    const F wii = w[3 * I + I], wjj = w[3 * J + J], wij = w[3 * I + J], wji = w[3 * J + I];
    const F r = mk(0.5f * (wii.re + wjj.re), 0.5f * (wii.im - wjj.im));
    const F s = mk(0.5f * (wij.re - wji.re), 0.5f * (wij.im + wji.im));
    const float k2 = r.re * r.re + r.im * r.im + s.re * s.re + s.im * s.im;
    if (!(k2 > 0)) return;
    const float ik = rsqrtf(k2);
    const F a = r * ik, b = s * ik;
    F R00, R01, R10, R11;
    if (MODE == 0) {
        float y[4];
        su2_draw_f(beta23 * (k2 * ik), k0, k1, link, sweep, sub, y);
        const F Y00 = mk(y[0], y[3]), Y01 = mk(y[2], y[1]), Y10 = mk(-y[2], y[1]), Y11 = mk(y[0], -y[3]);
        const F nb = mk(-b.re, -b.im);
        R00 = cmac(cmul(Y00, conjg(a)), Y01, conjg(b));
        R01 = cmac(cmul(Y00, nb), Y01, a);
        R10 = cmac(cmul(Y10, conjg(a)), Y11, conjg(b));
        R11 = cmac(cmul(Y10, nb), Y11, a);
    } else {
        const F D00 = conjg(a), D01 = mk(-b.re, -b.im), D10 = conjg(b), D11 = a;
        R00 = cmac(cmul(D00, D00), D01, D10);
        R01 = cmac(cmul(D00, D01), D01, D11);
        R10 = cmac(cmul(D10, D00), D11, D10);
        R11 = cmac(cmul(D10, D01), D11, D11);
    }
    rot_rows<I, J>(w, R00, R01, R10, R11);
    rot_rows<I, J>(u, R00, R01, R10, R11);
}

// U32: an FP32 copy of rows 0,1 of every link ([mu][6][V]), read for the staples
// and kept up to date with the links this launch writes.
template <int MODE>
__global__ void __launch_bounds__(kWilsonThreads) k_wilson32(Lat d, double2* __restrict__ U, float2* __restrict__ U32,
                                                             int mu, int parity, float beta, uint32_t k0, uint32_t k1,
                                                             uint32_t sweep)
{
    const int h = blockIdx.x * blockDim.x + threadIdx.x;
    if (h >= (d.V >> 1)) return;
    const int hx = d.L[0] >> 1;
    int c[4];
    int r = h / hx;
    const int xh = h - r * hx;
    c[1] = r % d.L[1];
    r /= d.L[1];
    c[2] = r % d.L[2];
    c[3] = r / d.L[2];
    c[0] = 2 * xh + ((parity + c[1] + c[2] + c[3]) & 1);
    const int s = c[0] + d.stride[1] * c[1] + d.stride[2] * c[2] + d.stride[3] * c[3];
    const int V = d.V, ne = d.ne;
    cx<float> A[9], uf[9], w[9];
    {
        Lat d32 = d;
        d32.ne = 6;
        staple_sum<float>(d32, U32, mu, s, c, A);
    }
    // the link itself from the FP32 copy, row 2 rebuilt in FP32
    load3<float>(U32, V, 6, mu, s, uf);
    mm<float>(uf, A, w);
    const uint32_t link = (uint32_t)mu * (uint32_t)V + (uint32_t)s;
    const float beta23 = beta * (2.0f / 3.0f);
    subgroup32<MODE, 0, 1>(uf, w, beta23, k0, k1, link, sweep, 0);
    subgroup32<MODE, 0, 2>(uf, w, beta23, k0, k1, link, sweep, 1);
    subgroup32<MODE, 1, 2>(uf, w, beta23, k0, k1, link, sweep, 2);
    // back to FP64 and onto SU(3) there: the stored link is unitary to FP64 rounding
    C u[9];
#pragma unroll
    for (int e = 0; e < 6; e++) u[e] = mk((double)uf[e].re, (double)uf[e].im);
    orthonormal_rows01(u);
#pragma unroll
    for (int e = 0; e < 6; e++) {
        st<double>(U + (size_t)(mu * ne + e) * V + s, u[e]);
        U32[(size_t)(mu * 6 + e) * V + s] = make_float2((float)u[e].re, (float)u[e].im);
    }
    if (ne == 9) {
        complete_row2(u, u + 6);
#pragma unroll
        for (int e = 6; e < 9; e++) st<double>(U + (size_t)(mu * 9 + e) * V + s, u[e]);
    }
}

// the FP32 copy of rows 0,1 of every link
__global__ void k_links_to_fp32(Lat d, const double2* __restrict__ U, float2* __restrict__ U32)
{
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= d.V) return;
    for (int mu = 0; mu < 4; mu++)
#pragma unroll
        for (int e = 0; e < 6; e++) {
            const double2 v = U[(size_t)(mu * d.ne + e) * d.V + s];
            U32[(size_t)(mu * 6 + e) * d.V + s] = make_float2((float)v.x, (float)v.y);
        }
}

// ---------------------------------------------------------------- plaquette

// Per block: sum over its sites of sum_{mu<nu} Re Tr[U_mu(x) U_nu(x+mu) (U_nu(x) U_mu(x+nu))^dag].
__global__ void __launch_bounds__(kPlaqThreads) k_plaq_partial(Lat d, const double2* __restrict__ U,
                                                              double* __restrict__ part)
{
    double acc = 0;
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < d.V; s += gridDim.x * blockDim.x) {
        int c[4];
        site_coords(d, s, c);
        for (int mu = 0; mu < 3; mu++) {
            const int sp = site_shift(d, s, c[mu], mu, +1);
            for (int nu = mu + 1; nu < 4; nu++) {
                const int sn = site_shift(d, s, c[nu], nu, +1);
                C a[9], b[9], p1[9], p2[9];
                load3<double>(U, d.V, d.ne, mu, s, a);
                load3<double>(U, d.V, d.ne, nu, sp, b);
                mm<double>(a, b, p1);
                load3<double>(U, d.V, d.ne, nu, s, a);
                load3<double>(U, d.V, d.ne, mu, sn, b);
                mm<double>(a, b, p2);
#pragma unroll
                for (int e = 0; e < 9; e++) acc += p1[e].re * p2[e].re + p1[e].im * p2[e].im;
            }
        }
    }
    __shared__ double red[kPlaqThreads];
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int w = kPlaqThreads / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = red[0];
}

// out = (sum of the n partials in a fixed order) * scale
__global__ void __launch_bounds__(kPlaqThreads) k_plaq_final(int n, const double* __restrict__ part, double scale,
                                                            double* __restrict__ out)
{
    __shared__ double red[kPlaqThreads];
    double acc = 0;
    for (int i = threadIdx.x; i < n; i += kPlaqThreads) acc += part[i];
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int w = kPlaqThreads / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = red[0] * scale;
}

// U_mu(x) = 1 in every stored plane
__global__ void k_unit_links(Lat d, double2* __restrict__ U)
{
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= d.V) return;
    for (int mu = 0; mu < 4; mu++)
        for (int e = 0; e < d.ne; e++)
            U[(size_t)(mu * d.ne + e) * d.V + s] = make_double2((e == 0 || e == 4 || e == 8) ? 1.0 : 0.0, 0.0);
}

}  // namespace

void launch_unit_links(cudaStream_t s, const Lat& d, double2* U)
{
    k_unit_links<<<(unsigned)((d.V + 255) / 256), 256, 0, s>>>(d, U);
}

int plaquette_blocks(int V)
{
    const int nb = (V + kPlaqThreads - 1) / kPlaqThreads;
    return nb < kPlaqBlocks ? nb : kPlaqBlocks;
}

void launch_links_to_fp32(cudaStream_t s, const Lat& d, const double2* U, float2* U32)
{
    k_links_to_fp32<<<(unsigned)((d.V + 255) / 256), 256, 0, s>>>(d, U, U32);
}

void launch_links_to_fx(cudaStream_t s, const Lat& d, double2* U)
{
    longlong2* X = reinterpret_cast<longlong2*>(U);
    k_links_to_fx<<<(unsigned)((d.V + 127) / 128), 128, 0, s>>>(d, X, X);
}
void launch_links_from_fx(cudaStream_t s, const Lat& d, double2* U)
{
    k_links_from_fx<<<(unsigned)((d.V + 127) / 128), 128, 0, s>>>(d, reinterpret_cast<const longlong2*>(U), U);
}

void launch_wilson_fx(cudaStream_t s, const Lat& d, longlong2* UX, int mu, int parity, int overrelax, double beta,
                      unsigned long long seed, unsigned int sweep)
{
    const unsigned nb = (unsigned)((d.V / 2 + kWilsonThreads - 1) / kWilsonThreads);
    const uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
    if (overrelax)
        k_wilson_fx<1><<<nb, kWilsonThreads, 0, s>>>(d, UX, mu, parity, beta, k0, k1, sweep);
    else
        k_wilson_fx<0><<<nb, kWilsonThreads, 0, s>>>(d, UX, mu, parity, beta, k0, k1, sweep);
}

void launch_wilson(cudaStream_t s, const Lat& d, double2* U, float2* U32, int mu, int parity, int overrelax,
                   double beta, unsigned long long seed, unsigned int sweep, int precision)
{
    const unsigned nb = (unsigned)((d.V / 2 + kWilsonThreads - 1) / kWilsonThreads);
    const uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
    if (precision == 32) {
        if (overrelax)
            k_wilson32<1><<<nb, kWilsonThreads, 0, s>>>(d, U, U32, mu, parity, (float)beta, k0, k1, sweep);
        else
            k_wilson32<0><<<nb, kWilsonThreads, 0, s>>>(d, U, U32, mu, parity, (float)beta, k0, k1, sweep);
    } else if (overrelax) {
        k_wilson<1><<<nb, kWilsonThreads, 0, s>>>(d, U, mu, parity, beta, k0, k1, sweep);
    } else {
        k_wilson<0><<<nb, kWilsonThreads, 0, s>>>(d, U, mu, parity, beta, k0, k1, sweep);
    }
}

void launch_plaquette(cudaStream_t s, const Lat& d, const double2* U, double* part, double* out)
{
    const int nb = plaquette_blocks(d.V);
    k_plaq_partial<<<nb, kPlaqThreads, 0, s>>>(d, U, part);
    k_plaq_final<<<1, kPlaqThreads, 0, s>>>(nb, part, 1.0 / (18.0 * (double)d.V), out);
}

}  // namespace lgf
