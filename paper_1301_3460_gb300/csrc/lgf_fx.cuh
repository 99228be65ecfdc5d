// 64-bit fixed-point arithmetic of the FP64 iterations.
//
// GB300 issues 2 FP64 operations per clock and SM but 63 mad.wide.s32 (32 x 32
// -> 64 bits with a 64-bit accumulator; both measured on the device), and the
// entries of SU(3) matrices are bounded by 1.  The matrix products of the FP64
// iterations therefore run on 64-bit integers: links and G hold a real x as
// x 2^61 (range +-4, resolution 4.3e-19; FP64 resolves 1.1e-16 near 1), g as x 2^62.
//
// Digits.  A value is h 2^32 + l with h, l signed 32-bit digits, and is kept in
// memory as that pair (l in the low word, h in the high one: the plain integer
// plus its own bit 31 in the upper half), so that a loaded word needs no work to
// be multiplied.
//
// Products.  Every partial product of two digits is one signed mad.wide.s32.  A
// sum of products keeps two accumulators: hh = sum h h' and m = sum (h l' + l h'),
// three mad.wide.s32 per product; the term l l' is dropped.  With scales p and q
// of the factors the sum is (hh 2^64 + m 2^32) 2^-(p+q) and the dropped term at
// most 2^(62-p-q): 2^-61 for g times a link, 2^-59 for the second product of an
// update (whose left factor is kept at 2^-59, where it needs no shift), 2^-60 for
// a row rebuilt from two others; the error of an updated link is about 2e-18,
// that of the FP64 products 1e-16.  The accumulators stay within 64 bits: for
// rows of norm <= 1 the six digits h of a row sum to at most sqrt(6) 2^(p-32)
// and |l| <= 2^31, so |m| <= sqrt(6) (2^61 + 2^60) < 2^63 for p = 62, q = 61.
//
// Sums of packed anti-Hermitian parts use the grid 2^-58 (range +-32; eight links'
// parts reach 27.4); adding them is exact and needs no FP64 operation.
#pragma once
#include "lgf_common.cuh"

namespace lgf {

using fx = long long;
constexpr int kFxBits = 61;  // links, G: x 2^61
constexpr int kFxG = 62;     // g: x 2^62
constexpr int kFxSum = 58;   // anti-Hermitian parts, their sums, Re Tr: x 2^58

using cfx = cx<fx>;

// the two signed digits of a value
struct dig {
    int h, l;
};
struct cdig {
    dig re, im;
};

__host__ __device__ __forceinline__ dig digits(fx v)
{
    const unsigned lo = (unsigned)v;
    return dig{(int)(v >> 32) + (int)(lo >> 31), (int)lo};
}
__host__ __device__ __forceinline__ cdig digits(cfx v) { return cdig{digits(v.re), digits(v.im)}; }
__host__ __device__ __forceinline__ fx value(dig d) { return ((fx)d.h << 32) + d.l; }

// digit pairs in memory
__device__ __forceinline__ cdig unpack(longlong2 v)
{
    return cdig{dig{(int)(v.x >> 32), (int)v.x}, dig{(int)(v.y >> 32), (int)v.y}};
}
__device__ __forceinline__ fx word(dig d) { return ((fx)d.h << 32) | (unsigned)d.l; }
__device__ __forceinline__ cdig ldd(const longlong2* p) { return unpack(__ldg(p)); }
__device__ __forceinline__ void std_(longlong2* p, cdig v) { *p = make_longlong2(word(v.re), word(v.im)); }

// sum of products of digit pairs
struct facc {
    fx hh, m;
};
// (inline PTX: the compiler widens (long long)a * b to a 64 x 64-bit product when a
// and b come out of 64-bit words, twice the instructions of an update)
__host__ __device__ __forceinline__ fx mulw(int a, int b)
{
#ifdef __CUDA_ARCH__
    fx c;
    asm("mul.wide.s32 %0, %1, %2;" : "=l"(c) : "r"(a), "r"(b));
    return c;
#else
    return (fx)a * b;
#endif
}
__host__ __device__ __forceinline__ fx madw(int a, int b, fx c)
{
#ifdef __CUDA_ARCH__
    fx r;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
#else
    return (fx)((unsigned long long)((fx)a * b) + (unsigned long long)c);
#endif
}
__host__ __device__ __forceinline__ void fmac(facc& a, dig x, dig y)
{
    a.hh = madw(x.h, y.h, a.hh);
    a.m = madw(x.h, y.l, a.m);
    a.m = madw(x.l, y.h, a.m);
}
// the sum's first product, with the rounding term of fval<S>
template <int S> __host__ __device__ __forceinline__ facc fmul(dig x, dig y)
{
    const fx m = S == 0 ? mulw(x.h, y.l) : madw(x.h, y.l, 1ll << (31 - S));
    return facc{mulw(x.h, y.h), madw(x.l, y.h, m)};
}
// the sum's value 2^S (hh 2^32 + m) / 2^32, rounded to nearest (S = 0: without the
// rounding term and its bits, hh + floor(m / 2^32))
template <int S> __host__ __device__ __forceinline__ fx fval(facc a)
{
    if constexpr (S == 0) return a.hh + (a.m >> 32);
    else return (a.hh << S) + (a.m >> (32 - S));
}
// p - n (p holds the rounding term)
__host__ __device__ __forceinline__ facc fsub(facc p, facc n) { return facc{p.hh - n.hh, p.m - n.m}; }

// Complex products take three real ones: with bs = Re b + Im b,
//   a b:        Re = p - q, Im = r - p - q,  r = (Re a + Im a) bs
//   a conj(b):  Re = p + q, Im = p - q - r,  r = (Re a - Im a) bs
// (p = Re a Re b, q = Im a Im b; sums over the row inside each).  The sums of a
// row's entries obey the same bound as its six reals above.
struct cdig3 {
    dig re, im, s;
};
__device__ __forceinline__ cdig3 with_sum(cdig a) { return cdig3{a.re, a.im, digits(value(a.re) + value(a.im))}; }
__device__ __forceinline__ cdig3 with_diff(cdig a) { return cdig3{a.re, a.im, digits(value(a.re) - value(a.im))}; }
__device__ __forceinline__ cdig3 with_sum(cfx a) { return cdig3{digits(a.re), digits(a.im), digits(a.re + a.im)}; }
__device__ __forceinline__ cdig3 with_diff(cfx a) { return cdig3{digits(a.re), digits(a.im), digits(a.re - a.im)}; }

// row a of a left factor (three entries, sums) times column j of the 3x3 b
template <int S> __device__ __forceinline__ cfx fx_mul(const cdig3* a, const cdig3* b, int j)
{
    facc p = fmul<S>(a[0].re, b[j].re), q = fmul<0>(a[0].im, b[j].im), r = fmul<S>(a[0].s, b[j].s);
#pragma unroll
    for (int k = 1; k < 3; k++) {
        fmac(p, a[k].re, b[3 * k + j].re);
        fmac(q, a[k].im, b[3 * k + j].im);
        fmac(r, a[k].s, b[3 * k + j].s);
    }
    if constexpr (S == 0) {
        const fx x = fval<0>(p), y = fval<0>(q);
        return cfx{x - y, fval<0>(r) - x - y};
    } else {
        return cfx{fval<S>(fsub(p, q)), fval<S>(facc{r.hh - p.hh - q.hh, r.m - p.m - q.m + (1ll << (31 - S))})};
    }
}

// row a (three entries, differences) times row j of conj(b): sum_k a_k conj(b_jk)
template <int S> __device__ __forceinline__ cfx fx_mul_dag(const cdig3* a, const cdig3* b, int j)
{
    facc p = fmul<S>(a[0].re, b[3 * j].re), q = fmul<0>(a[0].im, b[3 * j].im), r = fmul<0>(a[0].s, b[3 * j].s);
#pragma unroll
    for (int k = 1; k < 3; k++) {
        fmac(p, a[k].re, b[3 * j + k].re);
        fmac(q, a[k].im, b[3 * j + k].im);
        fmac(r, a[k].s, b[3 * j + k].s);
    }
    return cfx{fval<S>(facc{p.hh + q.hh, p.m + q.m}), fval<S>(facc{p.hh - q.hh - r.hh, p.m - q.m - r.m})};
}

// conj(a b - c d)
template <int S, typename D> __device__ __forceinline__ cfx fx_det2c(D a, D b, D c, D d)
{
    facc p = fmul<S>(a.re, b.re), n = fmul<0>(a.im, b.im), q = fmul<S>(c.re, d.im), o = fmul<0>(a.re, b.im);
    fmac(p, c.im, d.im);
    fmac(n, c.re, d.re);
    fmac(q, c.im, d.re);
    fmac(o, a.im, b.re);
    return cfx{fval<S>(fsub(p, n)), fval<S>(fsub(q, o))};
}

// third row of an SU(3) matrix, conj(row0 x row1); entry j
template <int S, typename D> __device__ __forceinline__ cfx fx_row2(const D* r0, const D* r1, int j)
{
    const int a = j == 0 ? 1 : j == 1 ? 2 : 0, b = j == 0 ? 2 : j == 1 ? 0 : 1;
    return fx_det2c<S>(r0[a], r1[b], r0[b], r1[a]);
}

__device__ __forceinline__ cfx ldx(const longlong2* p)
{
    const longlong2 v = __ldg(p);
    return cfx{v.x, v.y};
}
__device__ __forceinline__ void stx(longlong2* p, cfx v) { *p = make_longlong2(v.re, v.im); }

// ---------------------------------------------------------------- conversions

// x 2^Q of a double |x| < 2^(63-Q), rounded toward zero (exact for |x| >= 2^(53-Q)),
// by integer operations on the encoding: the mantissa at the
// top of a 64-bit word, shifted right by the exponent.  An infinite or NaN x sets
// *bad (the value is then not used).
template <int Q> __device__ __forceinline__ fx d2fx(double x, bool* bad)
{
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const int e = (int)((hi >> 20) & 0x7ffu);
    *bad = *bad || e == 0x7ff;
    const unsigned mh = 0x80000000u | ((hi & 0xfffffu) << 11) | (lo >> 21), ml = lo << 11;
    const unsigned long long m = ((unsigned long long)mh << 32) | ml;  // 1.0 -> 2^63
    int r = 1023 + 63 - Q - e;
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
