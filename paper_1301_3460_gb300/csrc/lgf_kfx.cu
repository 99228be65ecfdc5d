// The FP64 iterations on 64-bit fixed point: launchers of lgf_kfx.cuh and the g
// builders that store a fixed-point g.
#include "lgf_fxdiff.cuh"
#include "lgf_launch_impl.cuh"

namespace lgf {

namespace {
inline unsigned blocks(long n, int nt) { return (unsigned)((n + nt - 1) / nt); }
}  // namespace

cudaError_t fx_prepare(const Lat& d)
{
    int dev = 0, optin = 0;
    cudaError_t e;
    if ((e = cudaGetDevice(&dev))) return e;
    if ((e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev))) return e;
    if ((size_t)optin < plane_smem_bytes(d, sizeof(double2)) + 1024) return cudaErrorInvalidValue;
    if ((e = allow_max_smem(k_delta_fx<true, 32, double>, optin))) return e;
    if ((e = allow_max_smem(k_delta_fx<true, 128, double>, optin))) return e;
    if ((e = allow_max_smem(k_delta_fx<true, 32, float>, optin))) return e;
    if ((e = allow_max_smem(k_delta_fx<true, 128, float>, optin))) return e;
    if ((e = allow_max_smem(k_xyinv_g<double, fx, 32>, optin))) return e;
    if ((e = allow_max_smem(k_xyinv_g<double, fx, 128>, optin))) return e;
    if ((e = allow_max_smem(k_xyinv_g<float, fx, 32>, optin))) return e;
    if ((e = allow_max_smem(k_xyinv_g<float, fx, 128>, optin))) return e;
    if ((e = allow_max_smem(k_delta_fxt<32>, optin))) return e;
    if ((e = allow_max_smem(k_delta_fxt<128>, optin))) return e;
    if ((e = allow_max_smem(k_zt_fxt<32>, optin))) return e;
    if ((e = allow_max_smem(k_zt_fxt<128>, optin))) return e;
    if ((e = allow_max_smem(k_xyinv_fxt<32>, optin))) return e;
    if ((e = allow_max_smem(k_xyfwd_fxt<32>, optin))) return e;
    if ((e = allow_max_smem(k_xyfwd_fxt<128>, optin))) return e;
    if ((e = allow_max_smem(k_xyback_fxt<32>, optin))) return e;
    if ((e = allow_max_smem(k_xyback_fxt<128>, optin))) return e;
    return allow_max_smem(k_xyinv_fxt<128>, optin);
}

bool fxt_fits(const Lat& d, const Shape& sh) { return fxt_pencil_smem(d, sh.xw) <= 226 * 1024; }

size_t fxt_bytes(const Lat& d)
{
    return sizeof(FxExp) + (4 * (size_t)d.nplanes + 4 * (size_t)d.P + (size_t)d.P * d.L[2]) * sizeof(int) +
           (size_t)d.V * sizeof(fx) + (size_t)(d.L[0] + d.L[1] + d.L[2] + d.L[3]) * sizeof(longlong2);
}
FxtBuf fxt_carve(const Lat& d, void* p)
{
    FxtBuf b;
    b.tw = reinterpret_cast<longlong2*>(p);
    b.mx = reinterpret_cast<fx*>(b.tw + d.L[0] + d.L[1] + d.L[2] + d.L[3]);
    b.fe = reinterpret_cast<FxExp*>(b.mx + d.V);
    b.pexp = reinterpret_cast<int*>(b.fe + 1);
    b.bexp = b.pexp + 4 * (size_t)d.nplanes;
    b.me = b.bexp + 4 * (size_t)d.P;
    return b;
}
void launch_fxt_tables(const Lat& d, cudaStream_t s, const double* m64, const FxtBuf& b)
{
    k_make_mult_fx<<<blocks((long)d.P * d.L[2], 128), 128, 0, s>>>(d, m64, b.mx, b.me);
    k_make_roots_fx<<<1, 128, 0, s>>>(d, b.tw);
}
// threads: twice the shape's (its tiles were sized for FP64 lines in one thread), 512
// where one tile fills an SM's shared memory
static int fxt_threads(int nt, size_t smem, bool lines32)
{
    return !lines32 && smem > 113 * 1024 ? 512 : 2 * nt;
}

void launch_fxt_delta(const Lat& d, const Shape& sh, cudaStream_t s, const longlong2* AH, const fx* Fs, longlong2* Fd,
                      const FxtBuf& b, double* partials, Ctl* ctl, double2* hist, cudaGraphConditionalHandle h)
{
    const size_t sm = plane_smem_bytes(d, sizeof(longlong2));
    if (small_plane<double>(d))
        k_delta_fxt<32><<<d.nplanes, fxt_threads(sh.nt_xy, sm, true), sm, s>>>(d, AH, Fs, Fd, b.tw, b.pexp, b.fe, partials, ctl, hist, h);
    else
        k_delta_fxt<128><<<d.nplanes, fxt_threads(sh.nt_xy, sm, false), sm, s>>>(d, AH, Fs, Fd, b.tw, b.pexp, b.fe, partials, ctl, hist, h);
}
void launch_fxt_zt(const Lat& d, const Shape& sh, cudaStream_t s, longlong2* Fd, const FxtBuf& b, const Ctl* ctl, int nf, int own)
{
    const size_t sm = fxt_pencil_smem(d, sh.xw);
    const dim3 grid(d.L[0] / sh.xw, d.L[1], nf);
    if (short_zt_lines(d))
        k_zt_fxt<32><<<grid, fxt_threads(sh.nt_zt, sm, true), sm, s>>>(d, sh.xw, Fd, ctl, b.tw, b.mx, b.me, b.pexp, b.bexp, b.fe, own);
    else
        k_zt_fxt<128><<<grid, fxt_threads(sh.nt_zt, sm, false), sm, s>>>(d, sh.xw, Fd, ctl, b.tw, b.mx, b.me, b.pexp, b.bexp, b.fe, own);
}
void launch_fxt_xyinv_g(const Lat& d, const Shape& sh, cudaStream_t s, const longlong2* Fd, longlong2* g,
                        const FxtBuf& b, const Ctl* ctl, double2* Dt)
{
    const size_t sm = plane_smem_bytes(d, sizeof(longlong2));
    int xs = 0;
    while ((1 << xs) < sh.xw) xs++;
    if (small_plane<double>(d))
        k_xyinv_fxt<32><<<d.nplanes, fxt_threads(sh.nt_xy, sm, true), sm, s>>>(d, xs, Fd, g, ctl, b.tw, b.bexp, b.fe, Dt);
    else
        k_xyinv_fxt<128><<<d.nplanes, fxt_threads(sh.nt_xy, sm, false), sm, s>>>(d, xs, Fd, g, ctl, b.tw, b.bexp, b.fe, Dt);
}

void launch_fx_start(const Lat& d, cudaStream_t s, const longlong2* U64, longlong2* AH, fx* Fs, FxExp* fe)
{
    k_fx_start<<<blocks(d.V, 128), 128, 0, s>>>(d, U64, nullptr, AH, Fs, fe);
}
void launch_fx_start_bwd(const Lat& d, cudaStream_t s, const double2* U64, double2* Gud, longlong2* AH, fx* Fs, FxExp* fe)
{
    Lat dx = d;
    dx.nx = 9;  // the links on the grid wait in the slots of their cotangents
    k_fx_start<<<blocks(d.V, 128), 128, 0, s>>>(dx, reinterpret_cast<const longlong2*>(U64),
                                                reinterpret_cast<longlong2*>(Gud), AH, Fs, fe);
}
void launch_fx_enter(const Lat& d, cudaStream_t s, const longlong2* U64, const longlong2* G64, longlong2* U, longlong2* G,
                     Ctl* ctl)
{
    k_fx_enter<<<blocks(d.V, 128), 128, 0, s>>>(d, U64, G64, U, G, ctl);
}
void launch_fx_project(const Lat& d, cudaStream_t s, const float2* G32, double2* Gs, const double2* U64,
                       const double2* G64, longlong2* U, longlong2* G, longlong2* AH, fx* Fs, FxExp* fe, Ctl* ctl)
{
    k_switch_gs<<<blocks(d.V, 256), 256, 0, s>>>(d.V, G32, Gs, ctl);
    k_fx_project<<<blocks(d.V, 128), 128, 0, s>>>(d, U64, G64, Gs, U, G, AH, Fs, fe, ctl);
    k_phase_switch<<<1, 1, 0, s>>>(ctl);
}
void launch_fx_finish(const Lat& d, cudaStream_t s, const longlong2* U, const longlong2* G, double2* U64, double2* G64,
                      const Ctl* ctl)
{
    k_fx_finish<<<blocks(d.V, 128), 128, 0, s>>>(d, U, G, U64, G64, ctl);
}
void launch_fxt_accel(const Lat& d, const Shape& sh, cudaStream_t s, const double2* in, double2* out, longlong2* work,
                      int nf, const FxtBuf& b, const Ctl* ctl)
{
    const size_t sm = plane_smem_bytes(d, sizeof(longlong2));
    int xs = 0;
    while ((1 << xs) < sh.xw) xs++;
    const bool small = small_plane<double>(d);
    const int nt = fxt_threads(sh.nt_xy, sm, small);
    if (small)
        k_xyfwd_fxt<32><<<d.nplanes, nt, sm, s>>>(d, in, work, nf, b.tw, b.pexp, b.fe);
    else
        k_xyfwd_fxt<128><<<d.nplanes, nt, sm, s>>>(d, in, work, nf, b.tw, b.pexp, b.fe);
    launch_fxt_zt(d, sh, s, work, b, ctl, nf, 1);
    if (small)
        k_xyback_fxt<32><<<d.nplanes, nt, sm, s>>>(d, xs, work, out, nf, b.tw, b.bexp, b.fe);
    else
        k_xyback_fxt<128><<<d.nplanes, nt, sm, s>>>(d, xs, work, out, nf, b.tw, b.bexp, b.fe);
}
cudaError_t fxt_clear_bad(const FxtBuf& b, cudaStream_t s) { return cudaMemsetAsync(&b.fe->bad, 0, sizeof(int), s); }

void launch_fx_step_bwd(const Lat& d, cudaStream_t s, const longlong2* g, const double2* Fdt, double2* Gp, double2* Gud,
                        double2* Q, double alpha, double2* FA, double2* FB)
{
    k_bwd_update_fx<128, 3><<<dim3(blocks(d.V, 128), 4), 128, 0, s>>>(d, g, Gp, Gud, Q);
    k_bwd_reunit<<<blocks(d.V, 256), 256, 0, s>>>(d, Fdt, Gp, 4, 9, Q, alpha, FA, FB);
}

// A thread per link while its blocks of 32 sites, three to an SM, run in two rounds on the
// chip's 152 SMs.  With G, us a launch, a thread per link / per site: 4,096 sites 8.2 / 14.3,
// 8,192 10.2 / 14.3, 16,384 14.3 / 14.3, 20,736 15.4 / 18.4, 27,648 16.4 / 18.4, 32,768 19.5 to
// 20.5 / 18.4, 36,864 20.5 / 18.4, 49,152 26.6 / 24.6, 131,072 63.5 / 49.2.
constexpr int kUpdSmallV = 2 * 152 * 3 * 32;
template <int NX>
static void launch_fx_update_nx(const Lat& d, cudaStream_t s, longlong2* U, longlong2* G, const longlong2* g, Ctl* ctl,
                                longlong2* AH, fx* Fs)
{
    if (d.V <= kUpdSmallV)
        k_update_fx_small<NX><<<blocks(d.V, 32), kUpdSmallThreads, 0, s>>>(d, U, G, g, ctl, AH, Fs);
    else
        k_update_fx<NX><<<blocks(d.V, kUpdThreads), kUpdThreads, 0, s>>>(d, U, G, g, ctl, AH, Fs);
}
void launch_fx_update(const Lat& d, cudaStream_t s, longlong2* U, longlong2* G, const longlong2* g, Ctl* ctl,
                      longlong2* AH, fx* Fs)
{
    if (d.nx == 9)
        launch_fx_update_nx<9>(d, s, U, G, g, ctl, AH, Fs);
    else
        launch_fx_update_nx<6>(d, s, U, G, g, ctl, AH, Fs);
}

template <typename TF>
void launch_fx_delta(const Lat& d, const Shape& sh64, cudaStream_t s, const longlong2* AH, const fx* Fs,
                     vec2_t<TF>* Fd, double* partials, Ctl* ctl, double2* hist, bool fft, cudaGraphConditionalHandle h)
{
    const size_t sm = plane_smem_bytes(d, sizeof(vec2_t<TF>));
    if (!fft)
        k_delta_fx<false, 128, TF><<<d.nplanes, sh64.nt_xy, 0, s>>>(d, AH, Fs, Fd, partials, ctl, hist, h);
    else if (small_plane<double>(d))
        k_delta_fx<true, 32, TF><<<d.nplanes, sh64.nt_xy, sm, s>>>(d, AH, Fs, Fd, partials, ctl, hist, h);
    else
        k_delta_fx<true, 128, TF><<<d.nplanes, sh64.nt_xy, sm, s>>>(d, AH, Fs, Fd, partials, ctl, hist, h);
}

template <typename TF>
void launch_fx_xyinv_g(const Lat& d, const Shape& sh, cudaStream_t s, const vec2_t<TF>* Fd, longlong2* g,
                       const Ctl* ctl)
{
    const size_t sm = plane_smem_bytes(d, sizeof(vec2_t<TF>));
    if (small_plane<TF>(d))
        k_xyinv_g<TF, fx, 32><<<d.nplanes, sh.nt_xy, sm, s>>>(d, Fd, g, ctl);
    else
        k_xyinv_g<TF, fx, 128><<<d.nplanes, sh.nt_xy, sm, s>>>(d, Fd, g, ctl);
}

void launch_fx_build_g(const Lat& d, cudaStream_t s, const double2* Fd, longlong2* g, const Ctl* ctl)
{
    k_build_g<double, fx><<<blocks(d.V, 256), 256, 0, s>>>(d, Fd, g, ctl);
}

void launch_check_range(const Lat& d, cudaStream_t s, const double2* U64, int* wide)
{
    k_check_range<<<blocks(4L * d.V, 256), 256, 0, s>>>(d, U64, wide);
}

template void launch_fx_delta<double>(const Lat&, const Shape&, cudaStream_t, const longlong2*, const fx*, double2*,
                                      double*, Ctl*, double2*, bool, cudaGraphConditionalHandle);
template void launch_fx_delta<float>(const Lat&, const Shape&, cudaStream_t, const longlong2*, const fx*, float2*,
                                     double*, Ctl*, double2*, bool, cudaGraphConditionalHandle);
template void launch_fx_xyinv_g<double>(const Lat&, const Shape&, cudaStream_t, const double2*, longlong2*,
                                        const Ctl*);
template void launch_fx_xyinv_g<float>(const Lat&, const Shape&, cudaStream_t, const float2*, longlong2*, const Ctl*);

}  // namespace lgf
