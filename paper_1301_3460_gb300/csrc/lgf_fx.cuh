// 64-bit fixed-point arithmetic of the FP64 iterations.
//
// GB300 issues 2 FP64 operations per clock and SM but 63 mad.wide.s32 (32 x 32
// -> 64 bits with a 64-bit accumulator; both measured on the device), and the
// entries of SU(3) matrices are bounded by 1.  The matrix products of the FP64
// iterations therefore run on 64-bit integers: a real x is the integer
// x 2^61 (range +-4, resolution 4.3e-19; FP64 resolves 1.1e-16 near 1).
//
// Products.  v = h 2^32 + l with h, l signed 32-bit digits (l the low word read
// as signed, h the high word plus the low word's top bit), so every partial
// product is one signed mad.wide.s32.  A sum of products keeps two
// accumulators: hh = sum h h' and m = sum (h l' + l h'), three mad.wide.s32 per
// product; the term l l' 2^-122 is dropped (at most 2^-60, about 0.5e-18 rms:
// below FP64's own rounding of the same sum by a factor of about 50), and the
// result is hh 2^3 + round(m 2^-29).  For rows of norm <= 1 the accumulators
// stay within 64 bits: sum |h| over the six reals of a row is at most sqrt(6)
// 2^29 and |l| <= 2^31, so |m| <= 2 sqrt(6) 2^60 < 2^63.
//
// Sums of packed anti-Hermitian parts use a coarser grid, 2^-57 (range +-64, eight
// links' parts fit); adding them is exact and needs no FP64 operation.
#pragma once
#include "lgf_common.cuh"

namespace lgf {

using fx = long long;
constexpr int kFxBits = 61;   // matrices: x 2^61
constexpr int kFxSum = 57;    // anti-Hermitian parts, their sums, Re Tr: x 2^57

struct cfx {
    fx re, im;
};

// the two signed digits of a value
struct dig {
    int h, l;
};
struct cdig {
    dig re, im;
};

__device__ __forceinline__ dig digits(fx v)
{
    const unsigned lo = (unsigned)v;
    return dig{(int)(v >> 32) + (int)(lo >> 31), (int)lo};
}
__device__ __forceinline__ cdig digits(cfx v) { return cdig{digits(v.re), digits(v.im)}; }

// sum of products of digit pairs
struct facc {
    fx hh, m;
};
__device__ __forceinline__ fx madw(int a, int b, fx c)
{
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(c) : "r"(a), "r"(b));
    return c;
}
__device__ __forceinline__ void fmac(facc& a, dig x, dig y)
{
    a.hh = madw(x.h, y.h, a.hh);
    a.m = madw(x.h, y.l, a.m);
    a.m = madw(x.l, y.h, a.m);
}
__device__ __forceinline__ facc fzero() { return facc{0, 0}; }
__device__ __forceinline__ facc fround() { return facc{0, 1ll << 28}; }  // half a unit of the result
// the accumulator that continues -a (with the rounding term)
__device__ __forceinline__ facc fneg_round(facc a) { return facc{-a.hh, (1ll << 28) - a.m}; }
__device__ __forceinline__ fx fval(facc a) { return (a.hh << 3) + (a.m >> 29); }

// row i of a times the 3x3 b: out_j = sum_k a_k b_kj (digits of b row-major)
__device__ __forceinline__ void fx_row_mul(const cdig* a, const cdig* b, cfx* out)
{
#pragma unroll
    for (int j = 0; j < 3; j++) {
        facc n = fzero(), i = fround();
#pragma unroll
        for (int k = 0; k < 3; k++) {
            fmac(n, a[k].im, b[3 * k + j].im);
            fmac(i, a[k].re, b[3 * k + j].im);
            fmac(i, a[k].im, b[3 * k + j].re);
        }
        facc r = fneg_round(n);
#pragma unroll
        for (int k = 0; k < 3; k++) fmac(r, a[k].re, b[3 * k + j].re);
        out[j] = cfx{fval(r), fval(i)};
    }
}

// row a times b^dag: out_j = sum_k a_k conj(b_jk)
__device__ __forceinline__ void fx_row_mul_dag(const cdig* a, const cdig* b, cfx* out)
{
#pragma unroll
    for (int j = 0; j < 3; j++) {
        facc r = fround(), n = fzero();
#pragma unroll
        for (int k = 0; k < 3; k++) {
            fmac(r, a[k].re, b[3 * j + k].re);
            fmac(r, a[k].im, b[3 * j + k].im);
            fmac(n, a[k].re, b[3 * j + k].im);
        }
        facc i = fneg_round(n);
#pragma unroll
        for (int k = 0; k < 3; k++) fmac(i, a[k].im, b[3 * j + k].re);
        out[j] = cfx{fval(r), fval(i)};
    }
}

// conj(a b - c d)
__device__ __forceinline__ cfx fx_det2c(cdig a, cdig b, cdig c, cdig d)
{
    facc n = fzero();
    fmac(n, a.im, b.im);
    fmac(n, c.re, d.re);
    facc r = fneg_round(n);
    fmac(r, a.re, b.re);
    fmac(r, c.im, d.im);
    n = fzero();
    fmac(n, a.re, b.im);
    fmac(n, a.im, b.re);
    facc i = fneg_round(n);
    fmac(i, c.re, d.im);
    fmac(i, c.im, d.re);
    return cfx{fval(r), fval(i)};
}

// third row of an SU(3) matrix: conj(row0 x row1)
__device__ __forceinline__ void fx_row2(const cdig* r0, const cdig* r1, cfx* r2)
{
    r2[0] = fx_det2c(r0[1], r1[2], r0[2], r1[1]);
    r2[1] = fx_det2c(r0[2], r1[0], r0[0], r1[2]);
    r2[2] = fx_det2c(r0[0], r1[1], r0[1], r1[0]);
}

__device__ __forceinline__ cfx ldx(const longlong2* p)
{
    const longlong2 v = __ldg(p);
    return cfx{v.x, v.y};
}
__device__ __forceinline__ void stx(longlong2* p, cfx v) { *p = make_longlong2(v.re, v.im); }

// ---------------------------------------------------------------- conversions

// x 2^61 of a double |x| < 4, rounded toward zero (to the grid: 4.3e-19; exact
// for |x| >= 2^-8), by integer operations on the encoding: the mantissa at the
// top of a 64-bit word, shifted right by the exponent.  An infinite or NaN x sets
// *bad (the value is then not used).
__device__ __forceinline__ fx d2fx(double x, bool* bad)
{
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const int e = (int)((hi >> 20) & 0x7ffu);
    *bad = *bad || e == 0x7ff;
    const unsigned mh = 0x80000000u | ((hi & 0xfffffu) << 11) | (lo >> 21), ml = lo << 11;
    const unsigned long long m = ((unsigned long long)mh << 32) | ml;  // 1.0 -> 2^63
    int r = 1025 - e;  // 63 - 61 = 2 for e = 1023
    r = r > 63 ? 63 : (r < 0 ? 0 : r);
    unsigned long long v = m >> r;
    if (r == 63) v = 0;  // below the grid (zeros and subnormals among it)
    const fx s = -(fx)(hi >> 31);
    return ((fx)v ^ s) - s;
}

// the double nearest to v 2^-q
__device__ __forceinline__ double fx2d(fx v, int q)
{
    const double y = __ll2double_rn(v);
    const int hi = __double2hiint(y) - (q << 20);
    return v == 0 ? 0.0 : __hiloint2double(hi, __double2loint(y));
}

}  // namespace lgf
