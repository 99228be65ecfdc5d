// The 4D transform of the FP64 iterations on 64-bit integers: the same passes and
// tiles as k_delta, k_zt and k_xyinv_g (lgf_kernels.cuh), with block floating
// point in place of FP64.
//
// Every pass takes values of at most 2^B in magnitude, B = 62 - ceil(log2 L), so a
// line of L points cannot overflow, and its rounding errors (about one unit) are
// 2^-57 of the largest value for L = 32, below FP64's own (a line of 32 random
// values: 0.9 units rms against 58 for the FP64 codelet).  Between passes the
// values are shifted so that the largest fills B bits again: the bits in use are
// the OR of the values' magnitudes, gathered per tile in shared memory (per line
// for the accelerated t-lines, whose multipliers differ by orders of magnitude).
// A transform does not lower the largest value by more than half a bit, so after
// the first pass right shifts (rounded to nearest) are enough.  A value is
// the integer times 2^E; E is kept per xy-plane after the Delta kernel (pexp), per
// z,t pencil after the accelerator (bexp), and the consumer aligns them to the
// largest magnitude exponent of all planes (FxExp::amax1) or pencils (amax2).
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

// Right shift by r >= 0, rounded to nearest, ties away from zero: a tie rule that
// favours one sign would add up over the lattice into the lowest momenta, which
// the accelerator amplifies by up to p2max/p2min (at 64 x 16^3 ties up cost six times the
// error of an FP64 transform; this is below it).
struct RShift {
    fx rnd;
    int r;
};
__device__ __forceinline__ fx shift_round(fx v, fx rnd, int r) { return (v + rnd + (v >> 63)) >> r; }
__device__ __forceinline__ RShift rshift(int r)
{
    r = r < 0 ? 0 : (r > 62 ? 62 : r);
    return RShift{r > 0 ? 1ll << (r - 1) : 0ll, r};
}
__device__ __forceinline__ fx apply(RShift s, fx v) { return s.r ? shift_round(v, s.rnd, s.r) : v; }
__device__ __forceinline__ cfx apply(RShift s, cfx v) { return cfx{apply(s, v.re), apply(s, v.im)}; }
// The bits to reserve for values that are aligned to others before a pass over lines
// of L points: at least B + 1, so that the common exponent lies above every
// exponent and each alignment is a right shift of one bit or more.
__device__ __forceinline__ int align_top(unsigned o, int L) { return max(top_bits(o), fx_bits_rt(L) + 1); }
// the alignment: a right shift of the value's own by r >= 1
__device__ __forceinline__ cfx rshift1(cfx v, int r)
{
    r = r > 62 ? 62 : r;
    const fx rnd = 1ll << (r - 1);
    return cfx{shift_round(v.re, rnd, r), shift_round(v.im, rnd, r)};
}

// Delta (as k_delta_fx), theta and F, then the forward transform along x and y.
template <int LMAX>
__global__ void __launch_bounds__(kTileMaxThreads<double>, kTileMinBlocks<double, LMAX>) k_delta_fxt(
    Lat d, const longlong2* __restrict__ AH, const fx* __restrict__ Fs, longlong2* __restrict__ Fd,
    int* __restrict__ pexp, FxExp* fe, double* __restrict__ partials, Ctl* ctl, double2* hist)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    longlong2* sm = reinterpret_cast<longlong2*>(smem_raw);
    __shared__ unsigned s_or[3];
    if (ld_flag(&ctl->phase_done)) return;
    if (threadIdx.x < 3) s_or[threadIdx.x] = 0u;
    if (blockIdx.x == 0 && threadIdx.x == 0) fe->amax2 = kExpNone;
    __syncthreads();
    const int P = d.P, V = d.V, Lx = d.L[0], Ly = d.L[1];
    const int plane = blockIdx.x;
    const int s0 = plane * P;
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
    reduce_theta_F(th, fsum, partials, ctl, hist, V);
    __syncthreads();
    // x: to B bits (Delta shrinks by orders of magnitude over a fix: left shifts here)
    int E = -kFxSum;
    {
        const int sh = fx_bits_rt(Lx) - top_bits(s_or[0]);
        const int l = sh > 0 ? sh : 0;
        const RShift rs = rshift(-sh);
        E -= sh;
        o = 0;
        with_length<LMAX>(Lx, [&](auto Lc) {
            constexpr int L = decltype(Lc)::value;
            auto row = [&](int ln) {
                const int f = (int)fdiv((unsigned)ln, d.dLy), y = ln - f * Ly;
                return sm + f * fs + y * rsx;
            };
            lines_pass<fx, L, false>(
                4 * Ly,
                [&](int ln, int e) {
                    const cfx v = ldv<fx>(row(ln) + e);
                    return apply(rs, cfx{v.re << l, v.im << l});
                },
                [&](int ln, int e, cfx v) {
                    or_bits(o, v);
                    st<fx>(row(ln) + e, v);
                });
        });
        block_or(o, s_or + 1);
    }
    __syncthreads();
    {
        const RShift rs = rshift(top_bits(s_or[1]) - fx_bits_rt(Ly));
        E += rs.r;
        o = 0;
        longlong2* out = Fd + s0;
        with_length<LMAX>(Ly, [&](auto Lc) {
            constexpr int L = decltype(Lc)::value;
            lines_pass<fx, L, false>(
                4 * Lx,
                [&](int ln, int e) {
                    const int f = (int)fdiv((unsigned)ln, d.dLx), x = ln - f * Lx;
                    return apply(rs, ldv<fx>(sm + (f * fs + e * rsx + x)));
                },
                [&](int ln, int e, cfx v) {
                    const int f = (int)fdiv((unsigned)ln, d.dLx), x = ln - f * Lx;
                    or_bits(o, v);
                    st<fx>(out + (f * V + e * Lx + x), v);
                });
        });
        block_or(o, s_or + 2);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        pexp[plane] = E;
        atomicMax(&fe->amax1, E + align_top(s_or[2], d.L[2]));
    }
}

// z,t pencils (as k_zt): the multiplier p2max/(p2 V) of a t-line is kept as integers
// mx (digits, x 2^62) times 2^me, the largest of the line in [1/2, 1).
template <int LMAX>
__global__ void __launch_bounds__(kTileMaxThreads<double>, kTileMinBlocks<double, LMAX>) k_zt_fxt(
    Lat d, int xw, longlong2* __restrict__ Fd, const Ctl* ctl, const fx* __restrict__ mx, const int* __restrict__ me,
    const int* __restrict__ pexp, int* __restrict__ bexp, FxExp* fe)
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
    longlong2* g = Fd + (size_t)blockIdx.z * d.V + c0;
    fx* m64 = reinterpret_cast<fx*>(sm + Lt * rs);
    int* lexp = reinterpret_cast<int*>(m64 + xw * Lz * Lt);  // [kz][xi]
    if (threadIdx.x < 2) s_or[threadIdx.x] = 0u;
    if (threadIdx.x == 2) s_az = kExpNone;
    block_copy<8, fx>(
        xw * Lz * Lt,
        [&](int i) {
            const int zt = i >> xs, xi = i & (xw - 1);
            return __ldg(mx + c0 + (xi + P * zt));
        },
        [&](int i, fx v) { m64[i] = v; });
    __syncthreads();
    const int lane = (int)threadIdx.x & 31;
    // z forward: planes aligned to the largest
    const int Ez = __ldg(&fe->amax1) - fx_bits_rt(Lz);
    unsigned o = 0;
    with_length<LMAX>(Lz, [&](auto Lc) {
        constexpr int L = decltype(Lc)::value;
        lines_pass<fx, L, false>(
            xw * Lt,
            [&](int l, int e) {
                const int tt = l >> xs, xi = l & (xw - 1);
                const int p = e + L * tt;
                return rshift1(ldv<fx>(g + (xi + P * p)), Ez - __ldg(pexp + p));
            },
            [&](int l, int e, cfx v) {
                const int tt = l >> xs, xi = l & (xw - 1);
                or_bits(o, v);
                st<fx>(sm + tt * rs + e * xw + xi, v);
            });
    });
    block_or(o, s_or);
    __syncthreads();
    // t forward, accelerator, t inverse: lines (xi, kz), each with an exponent of its own
    {
        const RShift rt = rshift(top_bits(s_or[0]) - fx_bits_rt(Lt));
        const int Et = Ez + rt.r;
        int amax = kExpNone;
        with_length<LMAX>(Lt, [&](auto Lc) {
            constexpr int L = decltype(Lc)::value;
            constexpr int Tl = line_lanes<fx>(L), R = L / Tl, W = 32 / Tl, B = fx_bits(L);
            const int tau = lane / W, w = lane - tau * W;
            const int step = ((int)blockDim.x >> 5) * W, nlines = xw * Lz;
            for (int l0 = ((int)threadIdx.x >> 5) * W; l0 < nlines; l0 += step) {
                const int l = l0 + w;
                const bool ok = l < nlines;
                const int lc = ok ? l : l0;
                const int ml = __ldg(me + c0 + ((lc & (xw - 1)) + P * (lc >> xs)));
                cfx v[R];
#pragma unroll
                for (int j = 0; j < R; j++) v[j] = apply(rt, ldv<fx>(sm + line_pos_x<fx, L>(tau, j) * rs + lc));
                line_fwd<fx, L>(v, tau);
                unsigned b = 0;
#pragma unroll
                for (int r = 0; r < R; r++) {
                    const fx mw = m64[lc + xw * Lz * line_pos_k<fx, L>(tau, r)];
                    const dig m = dig{(int)(mw >> 32), (int)mw};
                    v[r] = cfx{xrmul(m, v[r].re), xrmul(m, v[r].im)};
                    or_bits(b, v[r]);
                }
#pragma unroll
                for (int h = 1; h < Tl; h <<= 1) b |= __shfl_xor_sync(0xffffffffu, b, h * W);
                const int sh = B - top_bits(b), sl = sh > 0 ? sh : 0;
                const RShift sr = rshift(-sh);
#pragma unroll
                for (int r = 0; r < R; r++) v[r] = apply(sr, cfx{v[r].re << sl, v[r].im << sl});
                line_inv<fx, L>(v, tau);
                b = 0;
#pragma unroll
                for (int j = 0; j < R; j++) or_bits(b, v[j]);
                const int El = Et + ml - sh;
                if (ok) {
#pragma unroll
                    for (int j = 0; j < R; j++) st<fx>(sm + line_pos_x<fx, L>(tau, j) * rs + l, v[j]);
                    if (tau == 0) lexp[l] = El;
                    amax = max(amax, El + align_top(b, Lz));
                }
            }
        });
        amax = __reduce_max_sync(0xffffffffu, amax);
        if (lane == 0) atomicMax(&s_az, amax);
    }
    __syncthreads();
    // z inverse, back to Fd
    {
        const int Eo = s_az - fx_bits_rt(Lz);
        o = 0;
        with_length<LMAX>(Lz, [&](auto Lc) {
            constexpr int L = decltype(Lc)::value;
            lines_pass<fx, L, true>(
                xw * Lt,
                [&](int l, int e) {
                    const int tt = l >> xs, xi = l & (xw - 1);
                    return rshift1(ldv<fx>(sm + tt * rs + e * xw + xi), Eo - lexp[e * xw + xi]);
                },
                [&](int l, int e, cfx v) {
                    const int tt = l >> xs, xi = l & (xw - 1);
                    or_bits(o, v);
                    st<fx>(g + (xi + P * (e + L * tt)), v);
                });
        });
        block_or(o, s_or + 1);
        __syncthreads();
        if (threadIdx.x == 0) {
            bexp[(blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] = Eo;
            atomicMax(&fe->amax2, Eo + align_top(s_or[1], d.L[1]));
        }
    }
}

// inverse along y and x, then g = reunit(1 + alpha/2 Delta~) in FP64, stored in fixed
// point.  xs: log2 of the pencils' width.
template <int LMAX>
__global__ void __launch_bounds__(kTileMaxThreads<double>, kTileMinBlocks<double, LMAX>) k_xyinv_fxt(
    Lat d, int xs, const longlong2* __restrict__ Fd, longlong2* __restrict__ g, const Ctl* ctl,
    const int* __restrict__ bexp, FxExp* fe)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    longlong2* sm = reinterpret_cast<longlong2*>(smem_raw);
    __shared__ unsigned s_or;
    if (ld_flag(&ctl->phase_done)) return;
    if (threadIdx.x == 0) s_or = 0u;
    if (blockIdx.x == 0 && threadIdx.x == 0) fe->amax1 = kExpNone;
    __syncthreads();
    const int P = d.P, V = d.V, Lx = d.L[0], Ly = d.L[1];
    const int s0 = blockIdx.x * P;
    const int rsx = plane_rsx(d), fs = plane_fs(d);
    const int nxc = Lx >> xs;
    int E = __ldg(&fe->amax2) - fx_bits_rt(Ly);
    unsigned o = 0;
    with_length<LMAX>(Ly, [&](auto Lc) {
        constexpr int L = decltype(Lc)::value;
        lines_pass<fx, L, true>(
            4 * Lx,
            [&](int l, int e) {
                const int f = (int)fdiv((unsigned)l, d.dLx), x = l - f * Lx;
                const int Eb = __ldg(bexp + (f * L + e) * nxc + (x >> xs));
                return rshift1(ldv<fx>(Fd + (s0 + f * V + e * Lx + x)), E - Eb);
            },
            [&](int l, int e, cfx v) {
                const int f = (int)fdiv((unsigned)l, d.dLx), x = l - f * Lx;
                or_bits(o, v);
                st<fx>(sm + (f * fs + e * rsx + x), v);
            });
    });
    block_or(o, &s_or);
    __syncthreads();
    const RShift rx = rshift(top_bits(s_or) - fx_bits_rt(Lx));
    E += rx.r;
    with_length<LMAX>(Lx, [&](auto Lc) {
        constexpr int L = decltype(Lc)::value;
        auto row = [&](int ln) {
            const int f = (int)fdiv((unsigned)ln, d.dLy), y = ln - f * Ly;
            return sm + f * fs + y * rsx;
        };
        lines_pass<fx, L, true>(
            4 * Ly, [&](int ln, int e) { return apply(rx, ldv<fx>(row(ln) + e)); },
            [&](int ln, int e, cfx v) { st<fx>(row(ln) + e, v); });
    });
    __syncthreads();
    // alpha/2 2^E (a field too large for FP64 gives infinity, as FP64 arithmetic does)
    const double h = scalbn(0.5 * ctl->alpha, E);
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

// the multipliers p2max/(p2(k) V) of every momentum as mx 2^(me - 62), me per t-line
// (one thread each), mx in digits
static __global__ void k_make_mult_fx(Lat d, const double* __restrict__ m64, fx* __restrict__ mx, int* __restrict__ me)
{
    const int nl = d.P * d.L[2];
    const int l = blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= nl) return;
    double top = 0.0;
    for (int t = 0; t < d.L[3]; t++) top = fmax(top, m64[l + nl * t]);
    const int e = ilogb(top) + 1;  // top 2^-e in [1/2, 1)
    me[l] = e;
    for (int t = 0; t < d.L[3]; t++) mx[l + nl * t] = word(digits(__double2ll_rn(scalbn(m64[l + nl * t], 62 - e))));
}

}  // namespace lgf
