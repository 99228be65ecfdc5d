// 64-bit fixed-point arithmetic of the FP64 iterations.
//
// GB300 issues 2 FP64 operations per clock and SM but 24 to 32 mad.wide.s32 (32 x 32
// -> 64 bits with a 64-bit accumulator, operands from distinct registers; both measured
// on the device), and the entries of SU(3) matrices are bounded by 1.  The matrix products of the FP64
// iterations therefore run on 64-bit integers: links and G hold a real x as
// x 2^61 (range +-4, resolution 4.3e-19; FP64 resolves 1.1e-16 near 1), g as x 2^62.
//
// Digits.  For products a value is split into h 2^32 + l with h, l signed 32-bit
// digits: l is the low word, h the high word plus the low word's top bit (one
// instruction).  Constant tables hold the pairs themselves.
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
// Sums of packed anti-Hermitian parts use the grid 2^-58 (range +-32); adding them is
// exact and needs no FP64 operation.  The largest entry of a part is 2 Im w00 - Im w11
// - Im w22: at most 2 sin a + 2 sin(a/2) = 3.520 (phases a = 1.872, -a/2, -a/2), so eight
// links reach 28.2.
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

// digit pairs in a table
__device__ __forceinline__ cdig unpack(longlong2 v)
{
    return cdig{dig{(int)(v.x >> 32), (int)v.x}, dig{(int)(v.y >> 32), (int)v.y}};
}
__device__ __forceinline__ fx word(dig d) { return ((fx)d.h << 32) | (unsigned)d.l; }
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
__host__ __device__ __forceinline__ facc fzero() { return facc{0, 0}; }
// p - n (p holds the rounding term)
__host__ __device__ __forceinline__ facc fsub(facc p, facc n) { return facc{p.hh - n.hh, p.m - n.m}; }

// Complex products take three real ones: with bs = Re b + Im b,
//   a b:        Re = p - q, Im = r - p - q,  r = (Re a + Im a) bs
//   a conj(b):  Re = p + q, Im = p - q - r,  r = (Re a - Im a) bs
// (p = Re a Re b, q = Im a Im b; sums over the row inside each).  The sums of a
// row's entries obey the same bound as its six reals above, so each of the three
// accumulators stays within 64 bits; their differences would not, and are taken
// between the rounded values.
struct cdig3 {
    dig re, im, s;
};
__device__ __forceinline__ cdig3 with_sum(cfx a) { return cdig3{digits(a.re), digits(a.im), digits(a.re + a.im)}; }
__device__ __forceinline__ cdig3 with_diff(cfx a) { return cdig3{digits(a.re), digits(a.im), digits(a.re - a.im)}; }

struct pqr {
    fx p, q, r;
};
// the three sums over a row a and three entries b[0], b[BS], b[2 BS], x 2^S
template <int S, int BS> __device__ __forceinline__ pqr fx_pqr(const cdig3* a, const cdig3* b)
{
    facc p = fmul<S>(a[0].re, b[0].re), q = fmul<S>(a[0].im, b[0].im), r = fmul<S>(a[0].s, b[0].s);
    // S = 0 rounds toward minus infinity; r starts low by half a unit, so that the
    // mean error of r - p - q is zero
    if constexpr (S == 0) r.m -= 1ll << 31;
#pragma unroll
    for (int k = 1; k < 3; k++) {
        fmac(p, a[k].re, b[BS * k].re);
        fmac(q, a[k].im, b[BS * k].im);
        fmac(r, a[k].s, b[BS * k].s);
    }
    return pqr{fval<S>(p), fval<S>(q), fval<S>(r)};
}
// row a of a left factor (three entries, sums) times column j of the 3x3 b
template <int S> __device__ __forceinline__ cfx fx_mul(const cdig3* a, const cdig3* b, int j)
{
    const pqr v = fx_pqr<S, 3>(a, b + j);
    return cfx{v.p - v.q, v.r - v.p - v.q};
}
// row a (three entries, differences) times row b of a conjugated factor
template <int S> __device__ __forceinline__ cfx fx_mul_dag(const cdig3* a, const cdig3* b)
{
    const pqr v = fx_pqr<S, 1>(a, b);
    return cfx{v.p + v.q, v.p - v.q - v.r};
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

// the double nearest to v 2^-q
__device__ __forceinline__ double fx2d(fx v, int q)
{
    const double y = __ll2double_rn(v);
    const int hi = __double2hiint(y) - (q << 20);
    return v == 0 ? 0.0 : __hiloint2double(hi, __double2loint(y));
}

// the same for any q, through zeros, subnormals and infinity where v 2^-q lies there
// (out of line: inlined, its FP64 operations are issued for every value)
static __device__ __noinline__ double fx2d_far(fx v, int q) { return scalbn(__ll2double_rn(v), -q); }
__device__ __forceinline__ double fx2d_safe(fx v, int q)
{
    const double y = __ll2double_rn(v);
    const int hi = __double2hiint(y), e = ((hi >> 20) & 0x7ff) - q;
    if (v == 0) return 0.0;
    if (e <= 0 || e >= 0x7ff) return fx2d_far(v, q);
    return __hiloint2double(hi - (q << 20), __double2loint(y));
}

// x 2^(60-e) of a double |x| < 2^e (e >= -1022), rounded toward zero; zero for what is not
// finite.  Subnormals count: no leading one, the exponent of the smallest normal numbers.
__device__ __forceinline__ fx d2fx_rel(double x, int e)
{
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const int ex = (int)((hi >> 20) & 0x7ffu);
    const unsigned mh = (ex ? 0x80000000u : 0u) | ((hi & 0xfffffu) << 11) | (lo >> 21), ml = lo << 11;
    const unsigned long long m = ((unsigned long long)mh << 32) | ml;  // 2^(ex-1023) -> 2^63
    const int r = 1023 + 3 + e - max(ex, 1);                           // 2^e -> 2^60
    unsigned long long v = (r >= 0 && r < 64) ? m >> r : 0ull;
    if (ex == 0x7ff) v = 0;
    const fx s = -(fx)(hi >> 31);
    return ((fx)v ^ s) - s;
}

// ---------------------------------------------------------------- Gram-Schmidt

// Rows 0,1 of g = reunit(X), X = 1 + A with A anti-Hermitian, on integers: X comes
// x 2^(61-q) with components below 2^(q-1) (2^60 as integers), the rows leave x 2^62.
// X X^dag = 1 + A A^dag, so both norms that are divided by are at least 1.  About 170
// mad.wide.s32 per site against 70 FP64 operations (2 per clock and SM); errors
// near 2^(q-60), FP64's 2^-53.

// sum of products with a run-time scale: 2^S (hh 2^32 + m) / 2^32, rounded
__device__ __forceinline__ fx fval_rt(facc a, int S) { return (a.hh << S) + ((a.m + (1ll << (31 - S))) >> (32 - S)); }

// |x|^2 of a row of three complex numbers (digits, x 2^(61-q)), x 2^(61-2q).  The
// squares of the low digits, dropped elsewhere, are added here to 15 bits: they are
// all positive, and a norm that is low at every site would shrink the links a
// little in every iteration.
__device__ __forceinline__ fx fx_norm2(const cdig* x)
{
    fx hh = 0, hl = 1ll << 27;
    unsigned ll = 0;
    auto add = [&](dig v) {
        hh = madw(v.h, v.h, hh);
        hl = madw(v.h, v.l, hl);
        const int t = v.l >> 17;
        ll += (unsigned)(t * t);
    };
#pragma unroll
    for (int j = 0; j < 3; j++) {
        add(x[j].re);
        add(x[j].im);
    }
    return (hh << 3) + ((hl + 2 * (fx)ll) >> 28);
}

// 1/sqrt(n) x 2^62 of n >= 1 given x 2^(61-2q), q <= 5: y0 from the FP32 reciprocal
// square root (22 bits), then one third-order step y0 (1 + d/2 + 3/8 d^2), d = 1 -
// n y0^2 (the binomial series of (1 - d)^(-1/2); next term 5/16 d^3 < 2^-62)
__device__ __forceinline__ fx fx_rsqrt(fx n, int q)
{
    const float nf = fmaf((float)(int)(n >> 32), 0x1p32f, (float)(unsigned)n) * __int_as_float((127 - 61 + 2 * q) << 23);
    const int y0 = __float2int_rn(rsqrtf(nf) * 0x1p30f);
    const dig nd = digits(n), yy = digits(mulw(y0, y0));  // y0^2 x 2^60
    // n y0^2 x 2^62: product x 2^(121-2q), all four partial products
    facc t = facc{mulw(nd.h, yy.h), madw(nd.h, yy.l, mulw(nd.l, yy.h))};
    t.m += mulw(nd.l, yy.l) >> 32;
    const fx d = (1ll << 62) - fval_rt(t, 5 + 2 * q);
    const int ds = (int)(d >> 12);  // x 2^50, |d| < 2^-20
    const fx c = (d >> 1) + ((mulw(ds, ds) >> 38) * 3 >> 3);
    const dig cd = digits(c);
    return ((fx)y0 << 32) + ((mulw(y0, cd.h) << 2) + (mulw(y0, cd.l) >> 30));
}

// r: rows 0,1 x 2^62, g: their digits
__device__ __forceinline__ void fx_gram_schmidt(const cfx* X, int q, cfx* r, cdig* g)
{
    cdig x0[3];
#pragma unroll
    for (int j = 0; j < 3; j++) x0[j] = digits(X[j]);
    const dig y = digits(fx_rsqrt(fx_norm2(x0), q));
    auto scale = [&](dig v, dig w) {  // x 2^(61-q) times x 2^62 -> x 2^62
        facc a = fzero();
        fmac(a, v, w);
        return fval_rt(a, 3 + q);
    };
#pragma unroll
    for (int j = 0; j < 3; j++) {
        r[j] = cfx{scale(x0[j].re, y), scale(x0[j].im, y)};
        g[j] = digits(r[j]);
    }
    // <r0, X1> = sum conj(r0_j) X1_j, x 2^(61-q)
    cdig x1[3];
#pragma unroll
    for (int j = 0; j < 3; j++) x1[j] = digits(X[3 + j]);
    facc pr = fmul<2>(x1[0].re, g[0].re), pi = fmul<2>(x1[0].im, g[0].re), n = fmul<0>(x1[0].re, g[0].im);
    fmac(pr, x1[0].im, g[0].im);
#pragma unroll
    for (int j = 1; j < 3; j++) {
        fmac(pr, x1[j].re, g[j].re);
        fmac(pi, x1[j].im, g[j].re);
        fmac(n, x1[j].re, g[j].im);
        fmac(pr, x1[j].im, g[j].im);
    }
    const cdig ip = digits(cfx{fval<2>(pr), fval<2>(fsub(pi, n))});
    // v = X1 - ip r0
    cdig v[3];
#pragma unroll
    for (int j = 0; j < 3; j++) {
        facc re = fmul<2>(ip.re, g[j].re), im = fmul<2>(ip.re, g[j].im), m = fmul<0>(ip.im, g[j].im);
        fmac(im, ip.im, g[j].re);
        v[j] = digits(cfx{X[3 + j].re - fval<2>(fsub(re, m)), X[3 + j].im - fval<2>(im)});
    }
    const dig z = digits(fx_rsqrt(fx_norm2(v), q));
#pragma unroll
    for (int j = 0; j < 3; j++) {
        r[3 + j] = cfx{scale(v[j].re, z), scale(v[j].im, z)};
        g[3 + j] = digits(r[3 + j]);
    }
}

// x 2^(61-q) of a float |x| < 2^(q-1), toward zero
__device__ __forceinline__ fx f2fx(float x, int q)
{
    const unsigned u = __float_as_uint(x);
    const int e = (int)((u >> 23) & 0xffu), r = e - 89 - q;  // 24-bit mantissa times 2^(e-150)
    const fx m = e ? (fx)((u & 0x7fffffu) | 0x800000u) : 0;
    const fx v = r >= 0 ? m << r : m >> (r < -63 ? 63 : -r);
    const fx s = -(fx)(u >> 31);
    return (v ^ s) - s;
}
// How far (x 2^62) an entry v of g may lie from the FP64 code's: the integer rows' error,
// about 2^-53, and 2^-46 of the entry or of the largest |alpha/2 Delta~| of the site (mx, x
// 2^(61-q)), eight times the FP64 code's bound.  The second is shifted down from where it
// stands: x 2^62 it does not fit a word from 2 on.
__host__ __device__ __forceinline__ unsigned long long g2f_tol(fx v, fx mx, int q)
{
    const fx a = (v < 0 ? -v : v) >> 46, b = mx >> (45 - q);
    return (unsigned long long)((1ll << (8 + q)) + (a > b ? a : b));
}
// The float nearest to v 2^-62.  *safe is cleared when a value within tol (x 2^62) of v
// may round to another float: v lies that close to the midpoint of two floats.
__device__ __forceinline__ float g2f(fx v, unsigned long long tol, bool* safe)
{
    const fx s = v >> 63;
    unsigned long long a = (unsigned long long)((v ^ s) - s);
    const int lz = __clzll((long long)a);
    if (lz > 40) {  // zero, or too few bits to tell
        *safe = false;
        return 0.f;
    }
    a <<= lz;
    // 24 leading bits kept, 40 dropped; distance of the dropped part from one half
    const long long d = (long long)(a & ((1ull << 40) - 1)) - (1ll << 39);
    const unsigned long long t = tol << lz;
    if ((unsigned long long)(d < 0 ? -d : d) <= t || (t >> lz) != tol) *safe = false;
    const unsigned m = (unsigned)(a >> 40) + (d > 0 ? 1u : 0u);  // 2^23 <= m <= 2^24
    const float f = (float)m * __int_as_float((127 - 22 - lz) << 23);
    return s ? -f : f;
}

// Rows 0,1 of g x 2^62 (r, digits rd) of FP32 fields alpha/2 Delta~ (packed as the
// transforms have them) of at most mx < 16 in magnitude; returns q.
__device__ __forceinline__ int fx_rows_of(float2 f0, float2 f1, float2 f2, float2 f3, float mx, cfx* r, cdig* rd)
{
    const int q = max(1, (int)(__float_as_uint(mx) >> 23) - 125);  // |v| < 2^(q-1)
    const fx one = 1ll << (61 - q);
    cfx X[6];
    X[0] = cfx{one, f2fx(f3.x, q)};
    X[1] = cfx{f2fx(f0.x, q), f2fx(f0.y, q)};
    X[2] = cfx{f2fx(f1.x, q), f2fx(f1.y, q)};
    X[3] = cfx{-X[1].re, X[1].im};  // -conj(Delta01)
    X[4] = cfx{one, f2fx(f3.y, q)};
    X[5] = cfx{f2fx(f2.x, q), f2fx(f2.y, q)};
    fx_gram_schmidt(X, q, r, rd);
    return q;
}
// The rows as the floats that the FP64 Gram-Schmidt of the same fields rounds to; false
// where that cannot be told.
__device__ __forceinline__ bool fx_rows_to_float(const cfx* r, float mx, int q, cx<float>* gs)
{
    bool safe = true;
    const fx m = f2fx(mx, q);
#pragma unroll
    for (int e = 0; e < 6; e++)
        gs[e] = cx<float>{g2f(r[e].re, g2f_tol(r[e].re, m, q), &safe), g2f(r[e].im, g2f_tol(r[e].im, m, q), &safe)};
    return safe;
}

// v x 2^62, |v| <= 1, rounded to the nearest double (ties to even), x 2^61: at most 53
// significant bits and none below 2^-61, so that the FP64 value is exact
__device__ __forceinline__ fx fx_round_double(fx v)
{
    const fx s = v >> 63;
    unsigned long long a = (unsigned long long)((v ^ s) - s);
    const int n = max(1, 11 - __clz((int)(a >> 32)));  // bits to drop, all in the low word
    a += (1u << (n - 1)) - 1u + (((unsigned)a >> n) & 1u);
    a = (a & ~(unsigned long long)((1u << n) - 1u)) >> 1;
    return ((fx)a ^ s) - s;
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

// The integer nearest to x 2^Q (ties to even, as __double2ll_rn(x 2^Q)) of a double |x| <
// 2^(62-Q); 0 for what is not finite.  The multiplication and conversion issue on the FP64
// pipe, two per clock and SM: a pass over the links of 32^4 takes 0.16 ms for them alone.
template <int Q> __device__ __forceinline__ fx d2fx_rn(double x)
{
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const int e = (int)((hi >> 20) & 0x7ffu);
    const unsigned mh = 0x80000000u | ((hi & 0xfffffu) << 11) | (lo >> 21), ml = lo << 11;
    const unsigned long long m = ((unsigned long long)mh << 32) | ml;  // 1.0 -> 2^63
    const int r = 1023 + 63 - Q - e;                                   // > 1; 64: x 2^Q in [1/2, 1)
    unsigned long long v = 0;
    if (r > 0 && r < 64) {
        const unsigned long long rest = m << (64 - r);  // the bits shifted out, one half at the top
        v = m >> r;
        v += rest > (1ull << 63) || (rest == (1ull << 63) && (v & 1)) ? 1 : 0;
    } else if (r == 64) {
        v = m > (1ull << 63) ? 1 : 0;
    }
    const fx s = -(fx)(hi >> 31);
    return ((fx)v ^ s) - s;
}

}  // namespace lgf
