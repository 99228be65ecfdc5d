// Host-side launch interface between the C ABI (lgf_capi.cu) and the kernel
// translation units (lgf_k64.cu: FP64 kernels and the conversion kernels,
// lgf_k32.cu: FP32 kernels, lgf_wilson.cu: configuration generation).  Splitting by precision keeps each unit small and
// lets them compile in parallel.
#pragma once
#include <cuda_runtime.h>

#include "lgf_common.cuh"

namespace lgf {

// per-axis twiddle tables exp(-2 pi i m / L_mu), momentum table 4 sin^2(pi k / L_mu)
struct Tables {
    const double2* tw64[4];
    const float2* tw32[4];
    const double* s2[4];
    double p2max;
    const double* mult64;  // p2max/(p2(k) V) per momentum (site-indexed)
    const float* mult32;
    const float* s2f;      // the four tables 4 sin^2(pi k / L_mu) in FP32, one after the other
};

// launch shape of the tiled FFT kernels of one precision
struct Shape {
    int nt_xy = 0;    // threads of the xy-plane kernels (a multiple of 32, at most 256)
    int nt_zt = 0;    // threads of the zt-pencil kernel (likewise)
    int xw = 0;       // x-columns per zt pencil (divides Lx)
    int zt_tma = 0;   // z,t kernel: 0 one block per pencil, 1 persistent with TMA-staged pencils
    int zt_grid = 0;  // blocks of the persistent form (zt_tma_grid)
};

// shared memory of the plane tile and of one pencil (element size elem)
size_t plane_tile_bytes(const Lat& d, size_t elem);
size_t pencil_tile_bytes(const Lat& d, int xw, size_t elem);
// shared-memory budget of one tile; extents whose tiles exceed it are refused
constexpr size_t kTileBudget = 220 * 1024;

template <typename T> cudaError_t prepare_kernels(const Lat& d, const Shape& sh);
template <typename T>
void launch_delta(const Lat& d, const Shape& sh, const Tables& tb, cudaStream_t s, const vec2_t<T>* AH, const T* Fs,
                  vec2_t<T>* Fd, double* partials, Ctl* ctl, double2* hist, bool fft);
template <typename T> void launch_ah_init(const Lat& d, cudaStream_t s, const vec2_t<T>* U, vec2_t<T>* AH, T* Fs);
template <typename T>
void launch_zt(const Lat& d, const Shape& sh, const Tables& tb, cudaStream_t s, vec2_t<T>* Fd, const Ctl* ctl);
// blocks of the TMA-staged z,t kernel for this lattice, nt threads and pencils
// of xw columns (0: the form cannot run that shape)
template <typename T> int zt_tma_grid(const Lat& d, int nt, int xw);
template <typename T>
void launch_xyinv_g(const Lat& d, const Shape& sh, const Tables& tb, cudaStream_t s, const vec2_t<T>* Fd,
                    vec2_t<T>* g, const Ctl* ctl);
template <typename T> void launch_build_g(const Lat& d, cudaStream_t s, const vec2_t<T>* Fd, vec2_t<T>* g, const Ctl* ctl);
template <typename T>
void launch_xy_fft(const Lat& d, const Shape& sh, const Tables& tb, cudaStream_t s, vec2_t<T>* Fd, bool inv);
template <typename T>
void launch_update(const Lat& d, cudaStream_t s, vec2_t<T>* U, vec2_t<T>* G, const vec2_t<T>* g, Ctl* ctl,
                   vec2_t<T>* AH, T* Fs);
// FP32 phase: the update fused with Delta, theta and F (links Uin -> Uout, Delta
// in space to Fd), and Delta, theta and F of stored links (every > 0: only on
// the FP32 phase's refresh iterations); grids of update_grid(V) blocks
int update_grid(int V);
void launch_update_delta32(const Lat& d, cudaStream_t s, const float2* Uin, float2* Uout, float2* G, const float2* g,
                           Ctl* ctl, float2* Fd, double* partials, double2* hist);
void launch_delta_links32(const Lat& d, cudaStream_t s, const float2* U, float2* Fd, double* partials, Ctl* ctl,
                          double2* hist, int every);

// FP32 phase: the g builder and the update in one persistent launch (k_gu); sync
// holds 4 + Lz Lt words, zeroed once before the first launch.  gu32_prepare
// raises the kernel's shared-memory limit.
cudaError_t gu32_prepare(const Lat& d);
void launch_gu32(const Lat& d, const Shape& sh, cudaStream_t s, const float2* Fd, float2* g, float2* U, float2* G,
                 float2* AH, float* Fs, Ctl* ctl, unsigned* sync);

// FP64 iterations with the accelerator in FP32 (FP64 unit): Delta, theta and F
// from the FP64 packed parts with the forward x,y transform in FP32 (Fd32), and
// the FP32 inverse x,y transform with the FP64 Gram-Schmidt writing an FP64 g;
// the FP32 z,t kernel (launch_zt<float>) sits between them
cudaError_t prepare_accel32(const Lat& d);
void launch_delta64_f32(const Lat& d, const Shape& sh64, cudaStream_t s, const double2* AH, const double* Fs,
                        float2* Fd, double* partials, Ctl* ctl, double2* hist);
void launch_xyinv_g32_64(const Lat& d, const Shape& sh32, cudaStream_t s, const float2* Fd, double2* g,
                         const Ctl* ctl);

// FP64 iterations on 64-bit fixed point (lgf_kfx.cuh): links and G on the grid 2^-61, g
// on 2^-62, packed parts and Re Tr on 2^-58.  start: parts and Re Tr of the stored
// links (start_bwd: and the links on the grid in the slots of their cotangents, for
// launch_fx_step_bwd); enter: the stored links (and G) to the grid, in place or elsewhere,
// when the loop goes on; project: the end of the FP32 phase (links rebuilt on the
// input's orbit, phase switched); finish: back to the stored FP64 links.  TF: precision
// of the transforms.  h: condition of the loop that the Delta kernel decides about (0: none).
struct FxExp;
// buffers of the integer transform (lgf_fxt.cuh): multipliers and exponents, carved
// from fxt_bytes(d) of device memory
struct FxtBuf {
    longlong2* tw = nullptr;  // [Lx + Ly + Lz + Lt] roots of unity
    long long* mx = nullptr;  // [V]
    FxExp* fe = nullptr;
    int* pexp = nullptr;      // [field][plane]
    int* bexp = nullptr;      // [field][pencil], at most 4 P
    int* me = nullptr;        // [t-lines]
};
size_t fxt_bytes(const Lat& d);
// whether a pencil of this shape fits into shared memory (the tile budget leaves no
// room for the lines' exponents in a few shapes of 16 columns)
bool fxt_fits(const Lat& d, const Shape& sh);
FxtBuf fxt_carve(const Lat& d, void* p);
void launch_fxt_tables(const Lat& d, cudaStream_t s, const double* m64, const FxtBuf& b);
cudaError_t fx_prepare(const Lat& d);
void launch_fx_start(const Lat& d, cudaStream_t s, const longlong2* U64, longlong2* AH, long long* Fs, FxExp* fe);
void launch_fx_start_bwd(const Lat& d, cudaStream_t s, const double2* U64, double2* Gud, longlong2* AH, long long* Fs,
                         FxExp* fe);
void launch_fx_enter(const Lat& d, cudaStream_t s, const longlong2* U64, const longlong2* G64, longlong2* U, longlong2* G,
                     Ctl* ctl);
void launch_fx_project(const Lat& d, cudaStream_t s, const float2* G32, double2* Gs, const double2* U64,
                       const double2* G64, longlong2* U, longlong2* G, longlong2* AH, long long* Fs, FxExp* fe, Ctl* ctl);
void launch_fx_finish(const Lat& d, cudaStream_t s, const longlong2* U, const longlong2* G, double2* U64, double2* G64,
                      const Ctl* ctl);
void launch_fx_update(const Lat& d, cudaStream_t s, longlong2* U, longlong2* G, const longlong2* g, Ctl* ctl,
                      longlong2* AH, long long* Fs);
template <typename TF>
void launch_fx_delta(const Lat& d, const Shape& sh64, cudaStream_t s, const longlong2* AH, const long long* Fs,
                     vec2_t<TF>* Fd, double* partials, Ctl* ctl, double2* hist, bool fft, cudaGraphConditionalHandle h);
template <typename TF>
void launch_fx_xyinv_g(const Lat& d, const Shape& sh, cudaStream_t s, const vec2_t<TF>* Fd, longlong2* g,
                       const Ctl* ctl);
// the iteration's transforms on integers: Delta + x,y forward; z,t with the
// multiplier (own: every field has exponents of its own); x,y inverse + g
void launch_fxt_delta(const Lat& d, const Shape& sh64, cudaStream_t s, const longlong2* AH, const long long* Fs,
                      longlong2* Fd, const FxtBuf& b, double* partials, Ctl* ctl, double2* hist,
                      cudaGraphConditionalHandle h);
void launch_fxt_zt(const Lat& d, const Shape& sh64, cudaStream_t s, longlong2* Fd, const FxtBuf& b, const Ctl* ctl,
                   int nf = 4, int own = 0);
void launch_fxt_xyinv_g(const Lat& d, const Shape& sh64, cudaStream_t s, const longlong2* Fd, longlong2* g,
                        const FxtBuf& b, const Ctl* ctl, double2* Dt = nullptr);
// the accelerator on nf packed FP64 fields (any values: a cotangent), in -> out, through
// the integer fields work; fxt_clear_bad before the first of several
cudaError_t fxt_clear_bad(const FxtBuf& b, cudaStream_t s);
void launch_fxt_accel(const Lat& d, const Shape& sh64, cudaStream_t s, const double2* in, double2* out, longlong2* work,
                      int nf, const FxtBuf& b, const Ctl* ctl);
// k_bwd_update on fixed point and the Gram-Schmidt's derivative; Gp is used up, Gud holds the
// links on entry
void launch_fx_step_bwd(const Lat& d, cudaStream_t s, const longlong2* g, const double2* Fdt, double2* Gp, double2* Gud,
                        double2* Q, double alpha, double2* FA, double2* FB);
void launch_fx_build_g(const Lat& d, cudaStream_t s, const double2* Fd, longlong2* g, const Ctl* ctl);
// *wide set when a stored link is not within 1e-3 of SU(3), or its stored row 2 not rows 0,1's
void launch_check_range(const Lat& d, cudaStream_t s, const double2* U64, int* wide);

// conversion, checking and mode-switch kernels (FP64 unit)
void launch_pack_links64(cudaStream_t s, int V, int ne, const double* in, double2* U, unsigned long long* err);
void launch_unpack_su3_64(cudaStream_t s, int V, int nmat, int ne, const double2* U, double* out);
void launch_identity_rows64(cudaStream_t s, int V, double2* G);
void launch_pack_delta(cudaStream_t s, int V, const double* in, double2* Fd);
void launch_unpack_delta(cudaStream_t s, int V, const double2* Fd, double* out);
void launch_unpack_full(cudaStream_t s, int V, const double2* g, double* out);
// n complex values FP64 -> FP32 and FP32 -> FP64, times scale
void launch_planes_to32(cudaStream_t s, long n, const double2* in, float2* out, double scale);
void launch_planes_to64(cudaStream_t s, long n, const float2* in, double2* out, double scale);
void launch_mixed_prep(cudaStream_t s, int V, int ne, const double2* U64, float2* U32, float2* G32, const Ctl* ctl);
void launch_switch(cudaStream_t s, const Lat& d, const float2* G32, double2* Gs, double2* U64, double2* G64,
                   Ctl* ctl);
void launch_loop_ctl(cudaStream_t s, Ctl* ctl, cudaGraphConditionalHandle h);
// FP32 phase: every `every` updates, G re-orthonormalised and U32 rebuilt as G U_in G^dag
void launch_refresh32(cudaStream_t s, const Lat& d32, int ne64, const double2* U64, float2* G32, float2* U32,
                      float2* AH32, float* Fs32, const Ctl* ctl, int every);
void launch_make_mult(cudaStream_t s, const Lat& d, const Tables& tb, double* m64, float* m32);
// derivative of one step and of the gluon propagator (lgf_diff.cuh)
void launch_g_from_dt(cudaStream_t s, int V, const double2* Fd, double2* g, double alpha);
void launch_pack_full(cudaStream_t s, int V, const double* in, double2* out);
void launch_unpack_planes(cudaStream_t s, int V, const double2* in, double* out);
void launch_step_bwd(cudaStream_t s, const Lat& d, const double2* U, const double2* g, const double2* Fdt,
                     double2* Gp, double2* Gud, double2* Ggs, double2* Q, double alpha, double2* FA, double2* FB);
void launch_bwd_delta(cudaStream_t s, const Lat& d, const double2* U, const double2* FA, const double2* FB,
                      const double2* Gud, double2* Gin);
int gluon_blocks(int V);
void launch_gluon(cudaStream_t s, const Lat& d, const double2* U, const Tables& tb, double2* part, double2* At,
                  double* D);
void launch_gluon_bwd(cudaStream_t s, const Lat& d, const double2* U, const double2* At, double coef, const Tables& tb,
                      double2* Gout);
// Wilson-action heat bath / overrelaxation of one (mu, parity) class of links,
// and the mean plaquette (lgf_wilson.cu)
void launch_wilson(cudaStream_t s, const Lat& d, double2* U, float2* U32, int mu, int parity, int overrelax,
                   double beta, unsigned long long seed, unsigned int sweep, int precision);
// the same on fixed-point links, converted once per call: [mu][9][V] from U on, where 36 V
// entries have to be free
void launch_links_to_fx(cudaStream_t s, const Lat& d, double2* U);
void launch_links_from_fx(cudaStream_t s, const Lat& d, double2* U);
void launch_wilson_fx(cudaStream_t s, const Lat& d, longlong2* UX, int mu, int parity, int overrelax, double beta,
                      unsigned long long seed, unsigned int sweep);
void launch_links_to_fp32(cudaStream_t s, const Lat& d, const double2* U, float2* U32);
void launch_unit_links(cudaStream_t s, const Lat& d, double2* U);
int plaquette_blocks(int V);
void launch_plaquette(cudaStream_t s, const Lat& d, const double2* U, double* part, double* out);
// writes the GPU's global nanosecond timer to *p
void launch_stamp(cudaStream_t s, unsigned long long* p);

}  // namespace lgf
