// The 4D transform of the FP64 iterations on 64-bit integers, in block floating point:
// Delta and the forward x,y transform per xy-plane, z,t with the accelerator per
// pencil, the inverse x,y transform and g per plane, each in a shared-memory tile as
// k_delta, k_zt and k_xyinv_g (lgf_kernels.cuh) do it in FP64.
//
// A line of L = A B points is transformed in two steps, A-point codelets with the
// twiddles w_L^(n2 k1) and B-point codelets (Cooley-Tukey: n = B n1 + n2, k = k1 +
// A k2), in place, so that a thread holds at most 8 complex integers (16 beyond 64
// points): 80 registers and 24 warps per SM, and 3 to 5 thousand instructions per
// kernel.  Whole 32-point lines in registers, as the FP64 kernels have them, take 168
// registers and 12,000 unrolled instructions in the z,t kernel and wait for
// instruction fetches.  32^4, Delta + x,y / z,t / x,y inverse + g: 372 / 426 / 379 us in
// FP64 (bound by the FP64 pipe), 178 / 220 / 215 us with whole integer lines, 136 / 124
// / 106 us like this (the last with the integer Gram-Schmidt, 174 us without).  What
// is left (ncu): Delta waits for its 32 loads per site (33% of the warps, issue 30%),
// z,t issues 44% of the time with 16 warps per SM (its tile and multipliers), the g
// builder 53%.
// In place, frequency k of a line lands on position (k mod A) B + k / A; the fields
// stay in that order between the kernels, the multiplier table is laid out in it,
// and the inverse (B-point, twiddles, A-point) takes it back.  An inverse runs the
// forward codelets with real and imaginary part exchanged on the way in and out.
//
// Every line transform takes values of at most 2^B in magnitude, B = 62 - ceil(log2
// L), so that L points cannot overflow, and its rounding errors (about one unit)
// are 2^-57 of the largest value for L = 32, below FP64's own (a line of 32 random
// values: 0.9 units rms against 58 for the FP64 codelet).  Between transforms the
// values are shifted so that the largest fills B bits again: the bits in use are
// the OR of the values' magnitudes, gathered per tile in shared memory (per line
// for the accelerated t-lines, whose multipliers differ by orders of magnitude).
// A transform does not lower the largest value by more than half a bit, so after
// the first one right shifts (rounded to nearest) are enough.  A value is
// the integer times 2^E; E is kept per xy-plane after the Delta kernel (pexp), per
// z,t pencil after the accelerator (bexp), and the consumer aligns them to the
// largest magnitude exponent of all planes (FxExp::amax1) or pencils (amax2).
// The fields of a Delta share their exponents (the first of each array): they end in one g
// on one grid, 2^-62, which is what a small field is known to there in any case.  The
// fields of a cotangent keep exponents of their own (OWN), as FP64 keeps their scales:
// colour components need not be of one size, and each ends in a gradient by itself.
// Field 3 stays at 3/2 of its value (lgf_kfx.cuh) through the transform.
#pragma once
#include "lgf_kfx.cuh"

namespace lgf {

__host__ __device__ constexpr int fx_bits(int L)  // B of a pass over lines of L points
{
    int c = 0;
    while ((1 << c) < L) c++;
    return 62 - c;
}
__device__ __forceinline__ int fx_bits_rt(int L) { return 62 - (32 - __clz(L - 1)); }

// OR of the magnitude bits of the high words
__device__ __forceinline__ void or_bits(unsigned& o, fx v)
{
    const int h = (int)(v >> 32);
    o |= (unsigned)(h ^ (h >> 31));
}
__device__ __forceinline__ void or_bits(unsigned& o, cfx v)
{
    or_bits(o, v.re);
    or_bits(o, v.im);
}
// every value is at most 2^top_bits in magnitude
__device__ __forceinline__ int top_bits(unsigned o) { return 64 - __clz(o | 1u) - (o == 0u ? 1 : 0); }

// the block's OR into *s (zeroed before, barrier after: the caller's)
__device__ __forceinline__ void block_or(unsigned o, unsigned* s)
{
    o = __reduce_or_sync(0xffffffffu, o);
    if ((threadIdx.x & 31) == 0 && o) atomicOr(s, o);
}

// OR into shared memory; the bits of most values are there after the first few
__device__ __forceinline__ void or_into(unsigned* s, unsigned b)
{
    if (b & ~*reinterpret_cast<volatile unsigned*>(s)) atomicOr(s, b);
}

// Right shift by r >= 1, rounded to nearest, ties away from zero: a tie rule that
// favours one sign would add up over the lattice into the lowest momenta, which
// the accelerator amplifies by up to p2max/p2min (error of the gauge transformation
// after a fix at 64 x 16^3: FP64 transforms 1.8e-16, ties up 4.3e-16, this 1.0e-16).
struct RShift {
    fx rnd;
    int r;
};
__device__ __forceinline__ RShift rshift(int r)
{
    r = r < 1 ? 1 : (r > 62 ? 62 : r);
    return RShift{1ll << (r - 1), r};
}
__device__ __forceinline__ fx apply(RShift s, fx v) { return (v + s.rnd + (v >> 63)) >> s.r; }
__device__ __forceinline__ cfx apply(RShift s, cfx v) { return cfx{apply(s, v.re), apply(s, v.im)}; }
// The bits to reserve for values that are aligned to others before a pass over lines
// of L points: at least B + 1, so that the common exponent lies above every
// exponent and each alignment is a right shift of one bit or more.
__device__ __forceinline__ int align_top(unsigned o, int L) { return max(top_bits(o), fx_bits_rt(L) + 1); }

// factors of a line length (B = 1: one codelet)
template <int L> struct Fac {
    static constexpr int A = L <= 8 ? L : L == 12 || L == 16 || L == 24 || L == 32 ? 4 : L == 48 || L == 64 ? 8 : 16;
    static constexpr int B = L / A;
};
__host__ __device__ inline int fac_a(int L) { return L <= 8 ? L : L <= 32 ? 4 : L <= 64 ? 8 : 16; }
// storage position of frequency k
__host__ __device__ inline int fac_pos(int k, int L) { return (k % fac_a(L)) * (L / fac_a(L)) + k / fac_a(L); }

// Blocks of up to 256 threads, three per SM (80 registers), for lines up to 32 points;
// longer lines (128 registers): up to 512 threads, which a tile too large for two
// blocks per SM gets.
template <int LMAX> constexpr int kFxtThreads = LMAX <= 32 ? 256 : 512;
template <int LMAX> constexpr int kFxtMinBlocks = LMAX <= 32 ? 3 : 1;

// One step over nlines lines: N-point codelets on the columns c = 0 .. NC-1 of each
// line, elements at positions c CS + i IS; with TW the results are multiplied by
// w^(c i) (tw: the length's roots).  ld(line) gives a functor position -> value,
// st(line) one (position, value); end(line, pos, v, N) sees a column's results first
// (pos(i): the position of the i-th).
// Consecutive threads take consecutive lines of one column.
template <int N, int NC, int CS, int IS, bool TW, typename LD, typename END, typename ST>
__device__ __forceinline__ void fx_step(int nlines, const longlong2* __restrict__ tw, LD ld, END end, ST st)
{
    const float inv = 1.0f / (float)nlines;
    const int n = NC * nlines;
#pragma unroll 1
    for (int i0 = threadIdx.x; i0 < n; i0 += blockDim.x) {
        // i0 / nlines, exact: (i0 + 1/2) / nlines is at least 1 / (2 nlines) from an integer
        const int c = NC == 1 ? 0 : (int)(((float)i0 + 0.5f) * inv), l = i0 - c * nlines;
        cfx v[N];
        auto get = ld(l);
#pragma unroll
        for (int i = 0; i < N; i++) v[i] = get(c * CS + i * IS);
        dft<fx, N, false>(v);
        if constexpr (TW) {
#pragma unroll
            for (int i = 1; i < N; i++) {
                const longlong2 w = __ldg(tw + c * i);
                const cdig d = unpack(w);
                v[i] = xcmul(d.re, d.im, digits(-value(d.im)), v[i]);
            }
        }
        end(l, [=](int i) { return c * CS + i * IS; }, v, std::integral_constant<int, N>{});
        auto put = st(l);
#pragma unroll
        for (int i = 0; i < N; i++) put(c * CS + i * IS, v[i]);
    }
}

struct NoEnd {
    template <typename POS, typename NN> __device__ __forceinline__ void operator()(int, POS, cfx*, NN) const {}
};

// A line transform (forward, or inverse when inv): first loads through ld, last
// stores through st after end, the values between the two steps in place through
// mid(line) -> pointer-like functors (mld, mst).
template <int LMAX, bool INV, typename LD, typename MLD, typename MST, typename END, typename ST>
__device__ __forceinline__ void fx_lines(int len, int nlines, const longlong2* __restrict__ tw, LD ld, MLD mld, MST mst,
                                         END end, ST st)
{
    with_length<LMAX>(len, [&](auto Lc) {
        constexpr int L = decltype(Lc)::value, A = Fac<L>::A, B = Fac<L>::B;
        if constexpr (B == 1) {
            fx_step<A, 1, 0, 1, false>(nlines, tw, ld, end, st);
        } else if constexpr (!INV) {
            fx_step<A, B, 1, B, true>(nlines, tw, ld, NoEnd{}, mst);
            __syncthreads();
            fx_step<B, A, B, 1, false>(nlines, tw, mld, end, st);
        } else {
            fx_step<B, A, B, 1, true>(nlines, tw, ld, NoEnd{}, mst);
            __syncthreads();
            fx_step<A, B, 1, B, false>(nlines, tw, mld, end, st);
        }
    });
}

__device__ __forceinline__ cfx swapped(longlong2 v) { return cfx{v.y, v.x}; }

// The shifts that bring values with the magnitude bits o to B + 1 bits before a shift by
// one (Delta shrinks by orders of magnitude over a fix: a left shift in the first pass):
// left by l, then right by r.
struct FwdShift {
    int l, r;
};
__device__ __forceinline__ FwdShift fwd_shift(unsigned o, int len)
{
    const int sh = fx_bits_rt(len) + 1 - top_bits(o);
    return FwdShift{sh > 0 ? sh : 0, sh < 0 ? 1 - sh : 1};
}

// The forward transform along x and y of nf fields of a plane in the tile to out.  s_or:
// [3][4] (a column per field, or the first for all): the values' bits before in the first
// row, zeros in the others; the results' bits in the last after the caller's next barrier.
template <int LMAX, bool OWN>
__device__ __forceinline__ void fx_plane_fwd(const Lat& d, longlong2* sm, longlong2* out, const longlong2* __restrict__ tw,
                                             unsigned* s_or, int nf)
{
    const int V = d.V, Lx = d.L[0], Ly = d.L[1];
    const int rsx = plane_rsx(d), fs = plane_fs(d);
#pragma unroll 1
    for (int pass = 0; pass < 2; pass++) {
        __syncthreads();
        // x rows, then y columns
        const int len = pass ? Ly : Lx, estr = pass ? rsx : 1;
        const FwdShift sh0 = fwd_shift(s_or[4 * pass], len);
        const RShift rs0 = rshift(sh0.r);
        unsigned o = 0;
        auto field = [&](int ln) { return (int)fdiv((unsigned)ln, pass ? d.dLx : d.dLy); };
        auto line = [&](int ln) {
            const int f = field(ln), c = ln - f * (pass ? Lx : Ly);
            return sm + f * fs + (pass ? c : c * rsx);
        };
        fx_lines<LMAX, false>(
            len, pass ? nf * Lx : nf * Ly, tw + (pass ? Lx : 0),
            [&](int ln) {
                const longlong2* p = line(ln);
                const FwdShift sh = OWN ? fwd_shift(s_or[4 * pass + field(ln)], len) : sh0;
                const RShift rs = OWN ? rshift(sh.r) : rs0;
                return [=](int e) {
                    const cfx v = ldv<fx>(p + e * estr);
                    return apply(rs, cfx{v.re << sh.l, v.im << sh.l});
                };
            },
            [&](int ln) {
                const longlong2* p = line(ln);
                return [=](int e) { return ldv<fx>(p + e * estr); };
            },
            [&](int ln) {
                longlong2* p = line(ln);
                return [=](int e, cfx v) { st<fx>(p + e * estr, v); };
            },
            [&](int ln, auto, const cfx* v, auto N) {
                if constexpr (OWN) o = 0;
#pragma unroll
                for (int j = 0; j < decltype(N)::value; j++) or_bits(o, v[j]);
                if constexpr (OWN) or_into(s_or + 4 * (pass + 1) + field(ln), o);
            },
            [&](int ln) {
                const int f = field(ln), c = ln - f * (pass ? Lx : Ly);
                longlong2* p = pass ? out + (f * V + c) : sm + f * fs + c * rsx;
                const int str = pass ? Lx : 1;
                return [=](int e, cfx v) { st<fx>(p + e * str, v); };
            });
        if constexpr (!OWN) block_or(o, s_or + 4 * (pass + 1));
    }
}
// Field f's exponent of a transformed plane into pexp and amax1: s_or the column of its bits,
// E its values' exponent before (after a barrier; a thread per field)
__device__ __forceinline__ void fx_plane_exp(const Lat& d, const unsigned* s_or, int f, int E, int plane,
                                             int* __restrict__ pexp, FxExp* fe)
{
    const FwdShift x = fwd_shift(s_or[0], d.L[0]), y = fwd_shift(s_or[4], d.L[1]);
    E += x.r - x.l + y.r - y.l;
    pexp[f * d.nplanes + plane] = E;
    atomicMax(&fe->amax1[f], E + align_top(s_or[8], d.L[2]));
}

// Delta (as k_delta_fx), theta and F, then the forward transform along x and y.
// tw: roots of unity of the four lengths, one after the other.
template <int LMAX>
__global__ void __launch_bounds__(kFxtThreads<LMAX>, kFxtMinBlocks<LMAX>) k_delta_fxt(
    Lat d, const longlong2* __restrict__ AH, const fx* __restrict__ Fs, longlong2* __restrict__ Fd,
    const longlong2* __restrict__ tw, int* __restrict__ pexp, FxExp* fe, double* __restrict__ partials, Ctl* ctl,
    double2* hist, cudaGraphConditionalHandle h)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    longlong2* sm = reinterpret_cast<longlong2*>(smem_raw);
    __shared__ unsigned s_or[12];
    if (ld_flag(&ctl->phase_done)) {
        end_loop(h);
        return;
    }
    if (threadIdx.x < 12) s_or[threadIdx.x] = 0u;
    if (blockIdx.x == 0 && threadIdx.x == 0) fe->amax2[0] = kExpNone;
    __syncthreads();
    const int P = d.P, V = d.V;
    const int plane = blockIdx.x;
    const int rsx = plane_rsx(d), fs = plane_fs(d);
    double th = 0.0, fsum = 0.0;
    unsigned o = 0;
    fx_delta_plane(d, AH, Fs, plane, th, fsum, [&](int xy, int x, int y, const cfx* raw, const cx<double>*) {
#pragma unroll
        for (int k = 0; k < 4; k++) {
            or_bits(o, raw[k]);
            st<fx>(sm + k * fs + y * rsx + x, raw[k]);
        }
    });
    block_or(o, s_or);
    reduce_theta_F(th, fsum, partials, ctl, hist, V, h);
    fx_plane_fwd<LMAX, false>(d, sm, Fd + plane * P, tw, s_or, 4);
    __syncthreads();
    if (threadIdx.x == 0) fx_plane_exp(d, s_or, 0, -kFxSum, plane, pexp, fe);
}

// z,t pencils (as k_zt): z forward, t forward and the accelerator, t inverse, z inverse
// in the tile [t][kz][xi].  The multiplier p2max/(p2 V) of a t-line is kept as
// integers mx (digits, x 2^62) times 2^me, the largest of the line in [1/2, 1); every
// accelerated t-line has an exponent of its own (lexp).  own: 1 for fields with exponents
// of their own, else 0.  Shared memory after the tile: the pencil's multipliers, lexp and
// the lines' magnitude bits [kz][xi].
inline size_t fxt_pencil_smem(const Lat& d, int xw)
{
    return pencil_smem_bytes(d, xw, sizeof(longlong2)) + (size_t)xw * d.L[2] * 2 * sizeof(int);
}

template <int LMAX>
__global__ void __launch_bounds__(kFxtThreads<LMAX>, kFxtMinBlocks<LMAX>) k_zt_fxt(
    Lat d, int xw, longlong2* __restrict__ Fd, const Ctl* ctl, const longlong2* __restrict__ tw,
    const fx* __restrict__ mx, const int* __restrict__ me, const int* __restrict__ pexp, int* __restrict__ bexp,
    FxExp* fe, int own)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    longlong2* sm = reinterpret_cast<longlong2*>(smem_raw);
    __shared__ unsigned s_or[2];
    __shared__ int s_az;
    if (ld_flag(&ctl->phase_done)) return;
    const int Lx = d.L[0], Lz = d.L[2], Lt = d.L[3], P = d.P;
    const int rs = pencil_rs(d, xw, sizeof(longlong2));
    const int xs = __ffs(xw) - 1;
    const int x0 = (int)blockIdx.x * xw, ky = (int)blockIdx.y;
    const int c0 = x0 + Lx * ky;
    const int fo = own * (int)blockIdx.z;
    longlong2* g = Fd + (size_t)blockIdx.z * d.V + c0;
    fx* m64 = reinterpret_cast<fx*>(sm + Lt * rs);
    int* lexp = reinterpret_cast<int*>(m64 + xw * Lz * Lt);       // [kz][xi]
    unsigned* lor = reinterpret_cast<unsigned*>(lexp + xw * Lz);  // [kz][xi]
    if (threadIdx.x < 2) s_or[threadIdx.x] = 0u;
    if (threadIdx.x == 2) s_az = kExpNone;
    for (int i = threadIdx.x; i < xw * Lz; i += blockDim.x) lor[i] = 0u;
    // the planes' values, aligned to B + 1 bits of the largest, and the multipliers
    int E = __ldg(fe->amax1 + fo) - fx_bits_rt(Lz) - 1;
    {
        const FastDiv dz = d.dLz;
        block_copy<4, longlong2>(
            xw * Lz * Lt, [&](int i) { return g[(i & (xw - 1)) + P * (i >> xs)]; },
            [&](int i, longlong2 v) {
                const int zt = i >> xs, t = (int)fdiv((unsigned)zt, dz), z = zt - t * Lz;
                const int r = E - __ldg(pexp + (fo * d.nplanes + zt));
                const cfx w = r > 0 ? apply(rshift(r), cfx{v.x, v.y}) : cfx{v.x, v.y};
                st<fx>(sm + t * rs + (z << xs) + (i & (xw - 1)), w);
            });
        block_copy<4, fx>(
            xw * Lz * Lt, [&](int i) { return __ldg(mx + c0 + ((i & (xw - 1)) + P * (i >> xs))); },
            [&](int i, fx v) { m64[i] = v; });
    }
    auto zline = [&](int l) { return sm + (l >> xs) * rs + (l & (xw - 1)); };
    auto tline = [&](int l) { return sm + l; };
    auto mload = [&](auto line, int str) {
        return [=](int l) {
            const longlong2* p = line(l);
            return [=](int e) { return ldv<fx>(p + e * str); };
        };
    };
    auto mstore = [&](auto line, int str) {
        return [=](int l) {
            longlong2* p = line(l);
            return [=](int e, cfx v) { st<fx>(p + e * str, v); };
        };
    };
    const longlong2 *twz = tw + d.L[0] + d.L[1], *twt = twz + Lz;
    // z forward
    unsigned o = 0;
    __syncthreads();
    {
        const RShift r1 = rshift(1);
        E += 1;
        fx_lines<LMAX, false>(
            Lz, xw * Lt, twz,
            [&](int l) {
                const longlong2* p = zline(l);
                return [=](int e) { return apply(r1, ldv<fx>(p + (e << xs))); };
            },
            mload(zline, xw), mstore(zline, xw),
            [&](int, auto, const cfx* v, auto N) {
#pragma unroll
                for (int j = 0; j < decltype(N)::value; j++) or_bits(o, v[j]);
            },
            mstore(zline, xw));
        block_or(o, s_or);
    }
    __syncthreads();
    // t forward and the multipliers (storage order: position by position)
    {
        const RShift rt = rshift(top_bits(s_or[0]) - fx_bits_rt(Lt));
        E += rt.r;
        fx_lines<LMAX, false>(
            Lt, xw * Lz, twt,
            [&](int l) {
                const longlong2* p = tline(l);
                return [=](int e) { return apply(rt, ldv<fx>(p + e * rs)); };
            },
            mload(tline, rs), mstore(tline, rs),
            [&](int l, auto pos, cfx* v, auto N) {
                const fx* mp = m64 + l;
                const int ms = xw * Lz;
                unsigned b = 0;
#pragma unroll
                for (int j = 0; j < decltype(N)::value; j++) {
                    const fx mw = mp[pos(j) * ms];
                    const dig m = dig{(int)(mw >> 32), (int)mw};
                    v[j] = cfx{xrmul(m, v[j].re), xrmul(m, v[j].im)};
                    or_bits(b, v[j]);
                }
                atomicOr(lor + l, b);
            },
            mstore(tline, rs));
    }
    __syncthreads();
    // t inverse, every line scaled to B bits by itself
    {
        int amax = kExpNone;
        const int B1 = fx_bits_rt(Lt) + 1;
        fx_lines<LMAX, true>(
            Lt, xw * Lz, twt,
            [&](int l) {
                const longlong2* p = tline(l);
                const int sh = B1 - top_bits(lor[l]), sl = sh > 0 ? sh : 0;
                const RShift r = rshift(1 - (sh < 0 ? sh : 0));
                return [=](int e) {
                    const cfx v = swapped(p[e * rs]);
                    return apply(r, cfx{v.re << sl, v.im << sl});
                };
            },
            mload(tline, rs), mstore(tline, rs),
            [&](int l, auto, const cfx* v, auto N) {
                unsigned b = 0;
#pragma unroll
                for (int j = 0; j < decltype(N)::value; j++) or_bits(b, v[j]);
                const int sh = B1 - top_bits(lor[l]);
                const int El = E + __ldg(me + c0 + ((l & (xw - 1)) + P * (l >> xs))) + 1 - sh;
                lexp[l] = El;
                amax = max(amax, El + align_top(b, Lz));
            },
            [&](int l) {
                longlong2* p = tline(l);
                return [=](int e, cfx v) { p[e * rs] = make_longlong2(v.im, v.re); };
            });
        amax = __reduce_max_sync(0xffffffffu, amax);
        if ((threadIdx.x & 31) == 0) atomicMax(&s_az, amax);
    }
    __syncthreads();
    // z inverse, back to Fd
    {
        E = s_az - fx_bits_rt(Lz);
        o = 0;
        fx_lines<LMAX, true>(
            Lz, xw * Lt, twz,
            [&](int l) {
                const longlong2* p = zline(l);
                const int* ep = lexp + (l & (xw - 1));
                return [=](int e) { return apply(rshift(E - ep[e << xs]), swapped(p[e << xs])); };
            },
            mload(zline, xw), mstore(zline, xw),
            [&](int, auto, const cfx* v, auto N) {
#pragma unroll
                for (int j = 0; j < decltype(N)::value; j++) or_bits(o, v[j]);
            },
            [&](int l) {
                longlong2* p = g + ((l & (xw - 1)) + P * Lz * (l >> xs));
                return [=](int e, cfx v) { p[e * P] = make_longlong2(v.im, v.re); };
            });
        block_or(o, s_or + 1);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        bexp[(blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] = E;
        atomicMax(&fe->amax2[fo], E + align_top(s_or[1], d.L[1]));
    }
}

// The inverse transform along y and x of nf fields of plane p into the tile.  Returns the
// exponent, or with OWN leaves the fields' in s_E; the values' bits in the second row of
// s_or ([2][4] as for fx_plane_fwd, zeroed on entry; barriers inside).
template <int LMAX, bool OWN>
__device__ __forceinline__ int fx_plane_inv(const Lat& d, int xs, const longlong2* __restrict__ Fd, longlong2* sm,
                                             const longlong2* __restrict__ tw, const int* __restrict__ bexp,
                                             const FxExp* fe, unsigned* s_or, int* s_E, int plane, int nf)
{
    const int P = d.P, V = d.V, Lx = d.L[0], Ly = d.L[1], s0 = plane * P;
    const int rsx = plane_rsx(d), fs = plane_fs(d);
    const int nxc = Lx >> xs;
    // the plane, aligned to B + 1 bits of the largest pencil: of each field, or of all
    int E = __ldg(fe->amax2) - fx_bits_rt(Ly) - 1;
    auto start = [&](int f) { return OWN ? __ldg(fe->amax2 + f) - fx_bits_rt(Ly) - 1 : E; };
    block_copy<4, longlong2>(
        nf * P,
        [&](int i) {
            const int f = (int)fdiv((unsigned)i, d.dP), xy = i - f * P;
            return Fd[s0 + f * V + xy];
        },
        [&](int i, longlong2 v) {
            const int f = (int)fdiv((unsigned)i, d.dP), xy = i - f * P, y = (int)fdiv((unsigned)xy, d.dLx), x = xy - y * Lx;
            const int r = start(f) - __ldg(bexp + (f * Ly + y) * nxc + (x >> xs));
            const cfx w = r > 0 ? apply(rshift(r), cfx{v.x, v.y}) : cfx{v.x, v.y};
            st<fx>(sm + (f * fs + y * rsx + x), w);
        });
#pragma unroll 1
    for (int pass = 0; pass < 2; pass++) {
        __syncthreads();
        // y columns, then x rows
        const int len = pass ? Lx : Ly, estr = pass ? 1 : rsx;
        auto shift = [&](int f) { return rshift(pass ? top_bits(s_or[OWN ? f : 0]) - fx_bits_rt(Lx) : 1); };
        const RShift rs0 = shift(0);
        if (!OWN) E += rs0.r;
        else if (pass && threadIdx.x < 4) s_E[threadIdx.x] = start((int)threadIdx.x) + 1 + shift((int)threadIdx.x).r;
        unsigned o = 0;
        auto field = [&](int ln) { return (int)fdiv((unsigned)ln, pass ? d.dLy : d.dLx); };
        auto line = [&](int ln) {
            const int f = field(ln), c = ln - f * (pass ? Ly : Lx);
            return sm + f * fs + (pass ? c * rsx : c);
        };
        fx_lines<LMAX, true>(
            len, pass ? nf * Ly : nf * Lx, tw + (pass ? 0 : Lx),
            [&](int ln) {
                const longlong2* p = line(ln);
                const RShift rs = OWN ? shift(field(ln)) : rs0;
                return [=](int e) { return apply(rs, swapped(p[e * estr])); };
            },
            [&](int ln) {
                const longlong2* p = line(ln);
                return [=](int e) { return ldv<fx>(p + e * estr); };
            },
            [&](int ln) {
                longlong2* p = line(ln);
                return [=](int e, cfx v) { st<fx>(p + e * estr, v); };
            },
            [&](int ln, auto, const cfx* v, auto N) {
                if constexpr (OWN) o = 0;
#pragma unroll
                for (int j = 0; j < decltype(N)::value; j++) or_bits(o, v[j]);
                if constexpr (OWN) or_into(s_or + 4 * pass + field(ln), o);
            },
            [&](int ln) {
                longlong2* p = line(ln);
                return [=](int e, cfx v) { p[e * estr] = make_longlong2(v.im, v.re); };
            });
        if constexpr (!OWN) block_or(o, s_or + 4 * pass);
    }
    __syncthreads();
    return E;
}

// inverse along y and x, then g = reunit(1 + alpha/2 Delta~) stored in fixed point, by
// the integer Gram-Schmidt (in FP64 where alpha/2 Delta~ exceeds 16: far beyond any
// step that converges).  xs: log2 of the pencils' width.  Dt (may be null) receives
// Delta~ itself, packed, in FP64.
template <int LMAX>
__global__ void __launch_bounds__(kFxtThreads<LMAX>, kFxtMinBlocks<LMAX>) k_xyinv_fxt(
    Lat d, int xs, const longlong2* __restrict__ Fd, longlong2* __restrict__ g, const Ctl* ctl,
    const longlong2* __restrict__ tw, const int* __restrict__ bexp, FxExp* fe, double2* __restrict__ Dt)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    longlong2* sm = reinterpret_cast<longlong2*>(smem_raw);
    __shared__ unsigned s_or[8];
    if (ld_flag(&ctl->phase_done)) return;
    if (threadIdx.x < 8) s_or[threadIdx.x] = 0u;
    if (blockIdx.x == 0 && threadIdx.x < 4) fe->amax1[threadIdx.x] = kExpNone;
    const int P = d.P, V = d.V, Lx = d.L[0];
    const int s0 = blockIdx.x * P;
    const int rsx = plane_rsx(d), fs = plane_fs(d);
    const int E = fx_plane_inv<LMAX, false>(d, xs, Fd, sm, tw, bexp, fe, s_or, nullptr, blockIdx.x, 4);
    if (Dt != nullptr)
        for (int xy = threadIdx.x; xy < P; xy += blockDim.x) {
            const int y = (int)fdiv((unsigned)xy, d.dLx), i = y * rsx + (xy - y * Lx);
#pragma unroll
            for (int f = 0; f < 4; f++) {
                const longlong2 v = sm[f * fs + i];
                const double k = f == 3 ? 2.0 / 3.0 : 1.0;
                Dt[(size_t)f * V + s0 + xy] = make_double2(fx2d(v.x, -E) * k, fx2d(v.y, -E) * k);
            }
        }
    // |alpha/2 Delta~| <= alpha/2 2^(E + top) < 2^(q-1); ha = alpha/2 = hm 2^(he-62) exactly
    const double ha = 0.5 * ctl->alpha;
    const int he = ilogb(ha) + 1;
    const int q = max(1, he + E + top_bits(s_or[4]) + 1);
    if (ha < 1e30 && q <= 5) {
        // X x 2^(61-q) = f hm 2^(he - 62 + E + 61 - q)
        const dig hm = digits(__double2ll_rn(scalbn(ha, 62 - he)));
        const dig hm3 = digits(__double2ll_rn(scalbn(ha * (2.0 / 3.0), 62 - he)));
        const int sh = he + E + 61 - q, sl = sh > 0 ? sh : 0;
        const RShift sr = rshift(-sh);
        const fx one = 1ll << (61 - q);
        auto scaled = [&](dig m, fx f) { return apply(sr, xrmul(m, f)); };
        auto scaledl = [&](dig m, fx f) { return xrmul(m, f) << sl; };
        for (int xy = threadIdx.x; xy < P; xy += blockDim.x) {
            const int y = (int)fdiv((unsigned)xy, d.dLx), x = xy - y * Lx;
            const int i = y * rsx + x;
            const cfx f0 = ldv<fx>(sm + i), f1 = ldv<fx>(sm + fs + i), f2 = ldv<fx>(sm + 2 * fs + i),
                      f3 = ldv<fx>(sm + 3 * fs + i);
            cfx X[6];
            if (sh < 0) {
                X[0] = cfx{one, scaled(hm3, f3.re)};
                X[1] = cfx{scaled(hm, f0.re), scaled(hm, f0.im)};
                X[2] = cfx{scaled(hm, f1.re), scaled(hm, f1.im)};
                X[4] = cfx{one, scaled(hm3, f3.im)};
                X[5] = cfx{scaled(hm, f2.re), scaled(hm, f2.im)};
            } else {
                X[0] = cfx{one, scaledl(hm3, f3.re)};
                X[1] = cfx{scaledl(hm, f0.re), scaledl(hm, f0.im)};
                X[2] = cfx{scaledl(hm, f1.re), scaledl(hm, f1.im)};
                X[4] = cfx{one, scaledl(hm3, f3.im)};
                X[5] = cfx{scaledl(hm, f2.re), scaledl(hm, f2.im)};
            }
            X[3] = cfx{-X[1].re, X[1].im};  // -conj(Delta01)
            cfx r[6];
            cdig rd[6];
            fx_gram_schmidt(X, q, r, rd);
#pragma unroll
            for (int e = 0; e < 6; e++) stx(g + (size_t)e * V + s0 + xy, r[e]);
#pragma unroll
            for (int j = 0; j < 3; j++) stx(g + (size_t)(6 + j) * V + s0 + xy, fx_row2<2>(rd, rd + 3, j));
        }
        return;
    }
    // a field too large for FP64 gives infinity, as FP64 arithmetic does
    const double h = scalbn(ha, E);
    const double h3 = h * (2.0 / 3.0);
    for (int xy = threadIdx.x; xy < P; xy += blockDim.x) {
        const int y = (int)fdiv((unsigned)xy, d.dLx), x = xy - y * Lx;
        const int i = y * rsx + x;
        const cfx f0 = ldv<fx>(sm + i), f1 = ldv<fx>(sm + fs + i), f2 = ldv<fx>(sm + 2 * fs + i),
                  f3 = ldv<fx>(sm + 3 * fs + i);
        cx<double> X[6], gm[6];
        const double a0 = h * __ll2double_rn(f0.re), a1 = h * __ll2double_rn(f0.im);
        X[0] = mk<double>(1.0, h3 * __ll2double_rn(f3.re));
        X[1] = mk<double>(a0, a1);
        X[2] = mk<double>(h * __ll2double_rn(f1.re), h * __ll2double_rn(f1.im));
        X[3] = mk<double>(-a0, a1);  // -conj(Delta01)
        X[4] = mk<double>(1.0, h3 * __ll2double_rn(f3.im));
        X[5] = mk<double>(h * __ll2double_rn(f2.re), h * __ll2double_rn(f2.im));
        gram_schmidt01(X, gm);
        store_g<fx>(g, V, s0 + xy, gm, ctl);
    }
}

// ---------------------------------------------------------------- FP64 fields through the transform

// The accelerator on nf packed fields in FP64 that are not a Delta (a cotangent): to
// integers relative to each field's largest value in the plane and forward along x and y; after
// k_zt_fxt, back.  A value that is not finite sets *bad, which makes every result NaN,
// as an FP64 transform would.
template <int LMAX>
__global__ void __launch_bounds__(kFxtThreads<LMAX>, kFxtMinBlocks<LMAX>) k_xyfwd_fxt(
    Lat d, const double2* __restrict__ in, longlong2* __restrict__ Fd, int nf, const longlong2* __restrict__ tw,
    int* __restrict__ pexp, FxExp* fe)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    longlong2* sm = reinterpret_cast<longlong2*>(smem_raw);
    __shared__ unsigned s_or[12], s_top[4];
    if (threadIdx.x < 12) s_or[threadIdx.x] = 0u;
    if (threadIdx.x < 4) s_top[threadIdx.x] = 0u;
    if (blockIdx.x == 0 && threadIdx.x < 4) fe->amax2[threadIdx.x] = kExpNone;
    __syncthreads();
    const int P = d.P, Lx = d.L[0], s0 = blockIdx.x * P;
    const int rsx = plane_rsx(d), fs = plane_fs(d);
    auto at = [&](int i) {
        const int f = (int)fdiv((unsigned)i, d.dP), xy = i - f * P, y = (int)fdiv((unsigned)xy, d.dLx);
        return f * fs + y * rsx + (xy - y * Lx);
    };
    // the doubles into the tile, each field's largest exponent
    block_copy<4, double2>(
        nf * P,
        [&](int i) {
            const int f = (int)fdiv((unsigned)i, d.dP);
            return __ldg(in + (size_t)f * d.V + s0 + (i - f * P));
        },
        [&](int i, double2 v) {
            unsigned* t = s_top + (int)fdiv((unsigned)i, d.dP);
            const unsigned top = max((unsigned)__double2hiint(v.x) & 0x7fffffffu, (unsigned)__double2hiint(v.y) & 0x7fffffffu);
            if (top > *reinterpret_cast<volatile unsigned*>(t)) atomicMax(t, top);
            reinterpret_cast<double2*>(sm)[at(i)] = v;
        });
    __syncthreads();
    auto exponent = [&](int f) { return (int)(s_top[f] >> 20) - 1022; };  // every |x| of the field < 2^e
    if (threadIdx.x < 4 && exponent((int)threadIdx.x) > 1024) fe->bad = 1;
    // x 2^(60-e) (a value in place of its double: the same thread, the same slot)
    for (int i = threadIdx.x; i < nf * P; i += blockDim.x) {
        const int f = (int)fdiv((unsigned)i, d.dP), e = exponent(f);
        const double2 v = reinterpret_cast<const double2*>(sm)[at(i)];
        const cfx w = cfx{d2fx_rel(v.x, e), d2fx_rel(v.y, e)};
        unsigned o = 0;
        or_bits(o, w);
        or_into(s_or + f, o);
        st<fx>(sm + at(i), w);
    }
    fx_plane_fwd<LMAX, true>(d, sm, Fd + s0, tw, s_or, nf);
    __syncthreads();
    if ((int)threadIdx.x < nf)
        fx_plane_exp(d, s_or + threadIdx.x, (int)threadIdx.x, exponent((int)threadIdx.x) - 60, blockIdx.x, pexp, fe);
}

template <int LMAX>
__global__ void __launch_bounds__(kFxtThreads<LMAX>, kFxtMinBlocks<LMAX>) k_xyback_fxt(
    Lat d, int xs, const longlong2* __restrict__ Fd, double2* __restrict__ out, int nf, const longlong2* __restrict__ tw,
    const int* __restrict__ bexp, FxExp* fe)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    longlong2* sm = reinterpret_cast<longlong2*>(smem_raw);
    __shared__ unsigned s_or[8];
    __shared__ int s_E[4];
    if (threadIdx.x < 8) s_or[threadIdx.x] = 0u;
    if (blockIdx.x == 0 && threadIdx.x < 4) fe->amax1[threadIdx.x] = kExpNone;
    const int P = d.P, Lx = d.L[0], s0 = blockIdx.x * P;
    const int rsx = plane_rsx(d), fs = plane_fs(d);
    fx_plane_inv<LMAX, true>(d, xs, Fd, sm, tw, bexp, fe, s_or, s_E, blockIdx.x, nf);
    const double nan = __hiloint2double(0x7ff80000, 0);
    const bool bad = ld_flag(&fe->bad) != 0;
    for (int i = threadIdx.x; i < nf * P; i += blockDim.x) {
        const int f = (int)fdiv((unsigned)i, d.dP), xy = i - f * P, y = (int)fdiv((unsigned)xy, d.dLx);
        const longlong2 v = sm[f * fs + y * rsx + (xy - y * Lx)];
        out[(size_t)f * d.V + s0 + xy] = bad ? make_double2(nan, nan) : make_double2(fx2d_safe(v.x, -s_E[f]), fx2d_safe(v.y, -s_E[f]));
    }
}

// the multipliers p2max/(p2(k) V) of every momentum as mx 2^(me - 62), me per t-line
// (one thread each), mx in digits; both in the storage order of the transform
static __global__ void k_make_mult_fx(Lat d, const double* __restrict__ m64, fx* __restrict__ mx, int* __restrict__ me)
{
    const int nl = d.P * d.L[2];
    const int l = blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= nl) return;
    double top = 0.0;
    for (int t = 0; t < d.L[3]; t++) top = fmax(top, m64[l + nl * t]);
    const int e = ilogb(top) + 1;  // top 2^-e in [1/2, 1)
    int c[4];
    site_coords(d, l, c);
    const int q = fac_pos(c[0], d.L[0]) + d.L[0] * (fac_pos(c[1], d.L[1]) + d.L[1] * fac_pos(c[2], d.L[2]));
    me[q] = e;
    for (int t = 0; t < d.L[3]; t++)
        mx[q + nl * fac_pos(t, d.L[3])] = word(digits(__double2ll_rn(scalbn(m64[l + nl * t], 62 - e))));
}

// roots of unity exp(-2 pi i m / L_mu), x 2^62 in digits, of the four lengths
static __global__ void k_make_roots_fx(Lat d, longlong2* __restrict__ tw)
{
    for (int mu = 0; mu < 4; mu++) {
        const int L = d.L[mu], step = 384 / L;
        for (int m = threadIdx.x; m < L; m += blockDim.x) {
            const cfx w = cfx{cos384x(m * step), -sin384x(m * step)};
            tw[m] = make_longlong2(word(digits(w.re)), word(digits(w.im)));
        }
        tw += L;
    }
}

}  // namespace lgf
