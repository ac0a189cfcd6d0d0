// Host-side launch wrappers of the device kernels (defined in
// pflbm_launch.cuh).  C is a population storage codec (PopPlain<float>,
// PopPlain<double>, PopDev<__half>, PopDev<__nv_bfloat16>); each is
// instantiated in a translation unit of its own (pflbm_f32.cu, pflbm_f64.cu,
// pflbm_f16.cu, pflbm_bf16.cu).  T-typed wrappers handle the planes kept in
// the arithmetic type (history, macroscopic fields, diagnostics).
#pragma once

#include <cuda_runtime.h>

#include "pflbm_kernels.cuh"
#include "pflbm_adjoint.cuh"
#include "pflbm_obstacle.cuh"

namespace pflbm {

template <class C>
cudaError_t launch_march(int model, int mode, const Phys<typename C::value_t>& P,
                         const Bufs<typename C::value_t>& B, cudaStream_t s);
// a pass (any mode) of the plain codecs, one node per thread; moments: keep the
// FP64 update's moment form
template <class C>
cudaError_t launch_tile(int model, int mode, const Phys<typename C::value_t>& P,
                        const Bufs<typename C::value_t>& B, bool unit_rates, bool moments, cudaStream_t s);
// TMA-staged steps of the 16-bit deviation codecs (they return
// cudaErrorNotSupported when the grid is too narrow; the caller then uses
// launch_march)
template <class C>
cudaError_t launch_step_tma(const Phys<typename C::value_t>& P, const Bufs<typename C::value_t>& B, int* err,
                            bool unit_rates, cudaStream_t s);
template <class C>
cudaError_t launch_step_tma_ch(const Phys<typename C::value_t>& P, const Bufs<typename C::value_t>& B, int* err,
                               bool unit_rates, cudaStream_t s);
// columns and rows of a block of the step with obstacles on the current device
template <class C>
void obs_step_grid(int nx, int ny, bool ch, int* bw, int* bh);
// deviation storage: pulled plane k of a set -> dense doubles of a region
template <class C>
cudaError_t launch_pull_export(const Phys<typename C::value_t>& P, const void* in, int set, int k, double* out,
                               double add, int x0, int y0, int w, int hgt, cudaStream_t s);
// deviation storage: pulled values (9 plain planes) -> encoded post-collision set
template <class C>
cudaError_t launch_restream(const Phys<typename C::value_t>& P, const typename C::value_t* in, void* out,
                            int set, cudaStream_t s);
template <typename T>
cudaError_t launch_pull(const Phys<T>& P, const T* in, T* out, cudaStream_t s);
template <typename T>
cudaError_t launch_unstream(const Phys<T>& P, const T* in, T* out, cudaStream_t s);
// plane k of a set of NP row-interleaved planes <-> dense doubles
template <typename T>
cudaError_t launch_export(const Phys<T>& P, const T* in, int NP, int k, double* out, double add,
                          int x0, int y0, int w, int hgt, cudaStream_t s);
template <typename T>
cudaError_t launch_import(const Phys<T>& P, const double* in, T* out, int NP, int k, double sub,
                          cudaStream_t s);
template <typename T>
cudaError_t launch_diag(const Phys<T>& P, const T* macro, const T* phi_prev, double* partial, int nparts,
                        const int* err, double* out, cudaStream_t s);
// solid obstacles (pflbm_obstacle.cuh): the reflecting links of every node
// from a dense byte mask, and one step (or MACRO / HIST / INIT pass) through
// the obstacle passes; phis, mus: one-plane work planes of the arithmetic
// type.  With use_tma the step runs on the tile (Allen-Cahn, plain storage) or
// TMA kernels (err: their time-out flag).  moments: as for launch_tile.
template <typename T>
cudaError_t launch_obs_links(const Phys<T>& P, const unsigned char* solid, uint16_t* obs, cudaStream_t s);
template <class C>
cudaError_t launch_obs(int model, int mode, const Phys<typename C::value_t>& P, const Bufs<typename C::value_t>& B,
                       typename C::value_t* phis, typename C::value_t* mus, bool unit_rates, bool moments,
                       int* err, bool use_tma, cudaStream_t s);
// discrete adjoint of the Allen-Cahn step (pflbm_adjoint.cuh), plain storage
template <typename T>
cudaError_t launch_adjoint_step(const Phys<T>& P, const void* state, long long pop_bytes, const AdjBufs& A,
                                double* gacc, bool hist_only, bool unit_rates, cudaStream_t s);
template <typename T>
long long adjoint_blocks(int nx, int ny);
template <typename T>
cudaError_t launch_adjoint_seed(const Phys<T>& P, const double* djdphi, const AdjBufs& A, cudaStream_t s);
template <typename T>
cudaError_t launch_adjoint_init(const Phys<T>& P, const AdjBufs& A, double* out, cudaStream_t s);

}  // namespace pflbm
