// Definitions of the launch wrappers declared in pflbm_launch.h.
#pragma once

#include <algorithm>

#include "pflbm_launch.h"

namespace pflbm {

template <class C, int MODEL>
static cudaError_t launch_march_model(int mode, const Phys<typename C::value_t>& P,
                                      const Bufs<typename C::value_t>& B, cudaStream_t s) {
  const dim3 grid((P.nx + BX - 1) / BX, (P.ny + LY - 1) / LY);
  switch (mode) {
    case MODE_STEP: k_march<C, MODEL, MODE_STEP><<<grid, BX, 0, s>>>(P, B); break;
    case MODE_MACRO: k_march<C, MODEL, MODE_MACRO><<<grid, BX, 0, s>>>(P, B); break;
    case MODE_HIST: k_march<C, MODEL, MODE_HIST><<<grid, BX, 0, s>>>(P, B); break;
    case MODE_INIT: k_march<C, MODEL, MODE_INIT><<<grid, BX, 0, s>>>(P, B); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

template <class C>
cudaError_t launch_march(int model, int mode, const Phys<typename C::value_t>& P,
                         const Bufs<typename C::value_t>& B, cudaStream_t s) {
  return model == MODEL_CH ? launch_march_model<C, MODEL_CH>(mode, P, B, s)
                           : launch_march_model<C, MODEL_AC>(mode, P, B, s);
}

// Number of SMs of the current device (looked up once per device).
static inline int device_sm_count() {
  static int sms[64] = {0};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) dev = 0;
  if (!sms[dev] && cudaDeviceGetAttribute(&sms[dev], cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    sms[dev] = 152;
  return sms[dev];
}

// Rows per block segment: LY, halved (down to 8) until the grid of strips of
// `tbx` columns holds at least `waves` waves of `per_sm` resident blocks, so
// that grids of a few million nodes still fill every SM.  Each segment
// re-forms two phi rows and re-stages its first rows, so long segments are
// kept wherever the grid is large enough.
static inline int segment_rows(int nx, int ny, int tbx, int per_sm, int waves = 2) {
  const long long target = (long long)waves * device_sm_count() * per_sm;
  const long long strips = (nx + tbx - 1) / tbx;
  int seg = LY;
  while (seg > 8 && strips * ((ny + seg - 1) / seg) < target) seg /= 2;
  return seg;
}

// Segment rows of the 16-bit Allen-Cahn TMA step (with or without
// obstacles): it is bound by instruction issue, so blocks of a partial wave
// run faster and one wave of blocks suffices.
template <class C>
static int tma_segment_rows(int nx, int ny) {
  using G = TmaCfg<C>;
  return segment_rows(nx, ny, G::TBX, G::threads / G::TBX, 1);
}

// Launch `kern` as a programmatic dependent of the kernel launched just
// before it on `s` (it may start once every block of that kernel has issued
// griddepcontrol.launch_dependents, and orders its reads of that kernel's
// output with griddepcontrol.wait), or as a plain launch.
template <typename... KArgs, typename... Args>
static cudaError_t launch_maybe_dependent(bool dependent, void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem,
                                          cudaStream_t s, Args... args) {
  if (!dependent) {
    kern<<<grid, block, smem, s>>>(args...);
    return cudaGetLastError();
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

// Tile of the one-node-per-thread pass; columns in equal strips of at most 32.
// FP32: 32 x 4 (4096^2: 522 us a step; 32 x 8 564, on one GPU); Cahn-Hilliard, whose ring is
// two nodes wide: 32 x 8.  FP64: 32 x 8, and on grids of
// few nodes 16 x 4 or 8 x 4, so that as many SMs as possible get nodes for
// their FP64 pipes (300 x 150: 26.7 us; 32 x 8 33.1).
template <class C>
static dim3 tile_shape(int nx, int ny, bool ch) {
  const bool fp64 = sizeof(typename C::value_t) == 8;
  const long long nodes = (long long)nx * ny, sms = device_sm_count();
  int t = fp64 ? (nodes < (1LL << 17) ? 64 : 256) : (ch ? 256 : 128);
  if (fp64 && nodes <= 64 * sms) t = 32;
  const int wide = t >= 128 ? 32 : (t == 64 ? 16 : 8);
  const int strips = (nx + wide - 1) / wide, bw = (nx + strips - 1) / strips;
  return dim3(bw, std::max(1, std::min(t / bw, ny)));
}

template <class C, int MODEL, int MODE, bool UR, bool OBS = false, bool MOM = sizeof(typename C::value_t) == 4>
static cudaError_t launch_tile_kernel(const Phys<typename C::value_t>& P, const Bufs<typename C::value_t>& B,
                                      cudaStream_t s) {
  using T = typename C::value_t;
  const dim3 b = tile_shape<C>(P.nx, P.ny, MODEL == MODEL_CH);
  constexpr int R = MODEL == MODEL_CH || OBS ? 2 : 1;
  size_t smem = sizeof(T) * (b.x + 2 * R) * (b.y + 2 * R);
  if (MODEL == MODEL_CH) smem += sizeof(T) * (b.x + 2) * (b.y + 2);
  const dim3 grid((P.nx + b.x - 1) / b.x, (P.ny + b.y - 1) / b.y);
  // A dependent launch places its blocks while the kernel before it still holds
  // SMs, and fills the idle ones unevenly.  FP64 blocks, which keep their SM's
  // pipe busy, then share SMs that others could relieve (128^2: 27 us a step
  // against 14.4), unless a block is one warp and every SM can take one.
  const bool dep = sizeof(T) == 4 || (b.x * b.y <= 32 && (long long)grid.x * grid.y <= device_sm_count());
  return launch_maybe_dependent(dep, k_tile<C, MODEL, MODE, UR, OBS, MOM>, grid, b, smem, s, P, B);
}

// FP64 Allen-Cahn runs with n_delta below its default keep the node update's
// moment form, operation for operation: the scheme amplifies rounding there (a
// one-ulp change of phi grows to 3e-3 in 2000 steps at n_delta = 3e-3, to 1e-14
// at the default 5e-3), so any other order of operations is another trajectory.
// With obstacles too (obs_ac).  Under 16 columns they relax all nine moments (UR =
// false), as the register-pipelined kernel that served such grids does: the 4 x 256
// channel at n_delta = 1e-5 amplifies rounding by up to 1e7 (node_update's form left
// it 4.9e-9 from where this one does).
template <class C>
static cudaError_t launch_tile_moments(int mode, const Phys<typename C::value_t>& P,
                                       const Bufs<typename C::value_t>& B, bool unit_rates, cudaStream_t s) {
  switch (mode) {
    case MODE_STEP:
      return unit_rates && P.nx >= 4 * XPAD ? launch_tile_kernel<C, MODEL_AC, MODE_STEP, true, false, true>(P, B, s)
                                            : launch_tile_kernel<C, MODEL_AC, MODE_STEP, false, false, true>(P, B, s);
    case MODE_MACRO: return launch_tile_kernel<C, MODEL_AC, MODE_MACRO, false, false, true>(P, B, s);
    case MODE_HIST: return launch_tile_kernel<C, MODEL_AC, MODE_HIST, false, false, true>(P, B, s);
    case MODE_INIT: return launch_tile_kernel<C, MODEL_AC, MODE_INIT, false, false, true>(P, B, s);
    default: return cudaErrorInvalidValue;
  }
}

template <class C, int MODEL>
static cudaError_t launch_tile_model(int mode, const Phys<typename C::value_t>& P,
                                     const Bufs<typename C::value_t>& B, bool unit_rates, cudaStream_t s) {
  switch (mode) {
    case MODE_STEP:
      return unit_rates ? launch_tile_kernel<C, MODEL, MODE_STEP, true>(P, B, s)
                        : launch_tile_kernel<C, MODEL, MODE_STEP, false>(P, B, s);
    case MODE_MACRO: return launch_tile_kernel<C, MODEL, MODE_MACRO, false>(P, B, s);
    case MODE_HIST: return launch_tile_kernel<C, MODEL, MODE_HIST, false>(P, B, s);
    case MODE_INIT: return launch_tile_kernel<C, MODEL, MODE_INIT, false>(P, B, s);
    default: return cudaErrorInvalidValue;
  }
}
template <class C>
cudaError_t launch_tile(int model, int mode, const Phys<typename C::value_t>& P,
                        const Bufs<typename C::value_t>& B, bool unit_rates, bool moments, cudaStream_t s) {
  if constexpr (sizeof(typename C::value_t) == 8)
    if (moments && model == MODEL_AC) return launch_tile_moments<C>(mode, P, B, unit_rates, s);
  return model == MODEL_CH ? launch_tile_model<C, MODEL_CH>(mode, P, B, unit_rates, s)
                           : launch_tile_model<C, MODEL_AC>(mode, P, B, unit_rates, s);
}

template <class C, bool UR, bool VSEG, bool OBS = false>
static cudaError_t launch_tma_seg(const Phys<typename C::value_t>& P, const Bufs<typename C::value_t>& B,
                                  int* err, cudaStream_t s, bool dependent = false) {
  using G = TmaCfg<C>;
  using L = TmaLayout<C, G::TBX, G::DF, G::DG>;
  // per function and device; cheap next to a step
  cudaError_t e = cudaFuncSetAttribute(k_step_tma<C, UR, VSEG, OBS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)L::bytes);
  if (e != cudaSuccess) return e;
  const dim3 grid((P.nx + G::TBX - 1) / G::TBX, (P.ny + P.seg_rows - 1) / P.seg_rows);
  // a programmatic dependent of the kernel before it: without obstacles the
  // previous step (its blocks start during that step's last blocks and wait
  // for it to finish), with obstacles the phi pass (the blocks away from the
  // obstacle start while the pass finishes; the near blocks wait for it
  // before reading its plane)
  return launch_maybe_dependent(!OBS || dependent, k_step_tma<C, UR, VSEG, OBS>, grid, dim3(G::TBX), L::bytes, s, P,
                                B, err);
}

// Segments of LY rows use the instantiation with the constant length (its
// register allocation is the tuned one); shorter ones the runtime-length one.
template <class C, bool UR, bool OBS = false>
static cudaError_t launch_tma_variant(const Phys<typename C::value_t>& P0, const Bufs<typename C::value_t>& B,
                                      int* err, cudaStream_t s, bool dependent = false) {
  Phys<typename C::value_t> P = P0;
  P.seg_rows = tma_segment_rows<C>(P.nx, P.ny);
  return P.seg_rows == LY ? launch_tma_seg<C, UR, false, OBS>(P, B, err, s, dependent)
                          : launch_tma_seg<C, UR, true, OBS>(P, B, err, s, dependent);
}

// Launch grid of the step with obstacles: columns and rows of a block.
template <class C>
static int tma_ch_segment_rows(int nx, int ny);
template <class C>
void obs_step_grid(int nx, int ny, bool ch, int* bw, int* bh) {
  if (ch) {
    *bw = TmaChCfg<C>::TBX;
    *bh = tma_ch_segment_rows<C>(nx, ny);
  } else if constexpr (C::dev) {
    *bw = TmaCfg<C>::TBX;
    *bh = tma_segment_rows<C>(nx, ny);
  } else {
    const dim3 b = tile_shape<C>(nx, ny, false);
    *bw = b.x;
    *bh = b.y;
  }
}

// Cahn-Hilliard step: same segment rule, its own launch shape (TmaChCfg).
template <class C>
static int tma_ch_segment_rows(int nx, int ny) {
  using G = TmaChCfg<C>;
  return segment_rows(nx, ny, G::TBX, G::threads / G::TBX);
}

template <class C, bool UR, bool VSEG, bool OBS = false>
static cudaError_t launch_tma_ch_seg(const Phys<typename C::value_t>& P, const Bufs<typename C::value_t>& B,
                                     int* err, cudaStream_t s, bool dependent = false) {
  using G = TmaChCfg<C>;
  using L = TmaChLayout<C, G::TBX, G::DF, G::DG>;
  cudaError_t e = cudaFuncSetAttribute(k_step_tma_ch<C, UR, VSEG, OBS>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::bytes);
  if (e != cudaSuccess) return e;
  const dim3 grid((P.nx + G::TBX - 1) / G::TBX, (P.ny + P.seg_rows - 1) / P.seg_rows);
  return launch_maybe_dependent(!OBS || dependent, k_step_tma_ch<C, UR, VSEG, OBS>, grid, dim3(G::TBX), L::bytes, s,
                                P, B, err);
}

template <class C>
cudaError_t launch_step_tma_ch(const Phys<typename C::value_t>& P0, const Bufs<typename C::value_t>& B, int* err,
                               bool unit_rates, cudaStream_t s) {
  if (P0.nx < 4 * XPAD) return cudaErrorNotSupported;
  Phys<typename C::value_t> P = P0;
  P.seg_rows = tma_ch_segment_rows<C>(P.nx, P.ny);
  if (P.seg_rows == LY)
    return unit_rates ? launch_tma_ch_seg<C, true, false>(P, B, err, s) : launch_tma_ch_seg<C, false, false>(P, B, err, s);
  return unit_rates ? launch_tma_ch_seg<C, true, true>(P, B, err, s) : launch_tma_ch_seg<C, false, true>(P, B, err, s);
}

// The launch shape per storage codec (strip width, staging depth, blocks
// per SM) and the measurements behind it are given with TmaCfg.
template <class C>
cudaError_t launch_step_tma(const Phys<typename C::value_t>& P, const Bufs<typename C::value_t>& B, int* err,
                            bool unit_rates, cudaStream_t s) {
  if (P.nx < 4 * XPAD) return cudaErrorNotSupported;
  return unit_rates ? launch_tma_variant<C, true>(P, B, err, s) : launch_tma_variant<C, false>(P, B, err, s);
}

static inline dim3 row_grid(int nx, int ny, int threads) { return dim3((nx + threads - 1) / threads, ny); }

template <class C>
cudaError_t launch_pull_export(const Phys<typename C::value_t>& P, const void* in, int set, int k, double* out,
                               double add, int x0, int y0, int w, int hgt, cudaStream_t s) {
  k_pull_export<C><<<row_grid(w, hgt, 128), 128, 0, s>>>(P, in, set, k, out, add, x0, y0, w, hgt);
  return cudaGetLastError();
}

template <class C>
cudaError_t launch_restream(const Phys<typename C::value_t>& P, const typename C::value_t* in, void* out,
                            int set, cudaStream_t s) {
  k_restream<C><<<row_grid(P.nx, P.ny, 128), 128, 0, s>>>(P, in, out, set);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_pull(const Phys<T>& P, const T* in, T* out, cudaStream_t s) {
  k_pull<T><<<row_grid(P.nx, P.ny, 128), 128, 0, s>>>(P, in, out);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_unstream(const Phys<T>& P, const T* in, T* out, cudaStream_t s) {
  k_unstream<T><<<row_grid(P.nx, P.ny, 128), 128, 0, s>>>(P, in, out);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_export(const Phys<T>& P, const T* in, int NP, int k, double* out, double add,
                          int x0, int y0, int w, int hgt, cudaStream_t s) {
  k_export<T><<<row_grid(w, hgt, 128), 128, 0, s>>>(P, in, NP, k, out, add, x0, y0, w, hgt);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_import(const Phys<T>& P, const double* in, T* out, int NP, int k, double sub,
                          cudaStream_t s) {
  k_import<T><<<row_grid(P.nx, P.ny, 128), 128, 0, s>>>(P, in, out, NP, k, sub);
  return cudaGetLastError();
}

// (each a programmatic dependent of the kernel before it)
template <typename T>
cudaError_t launch_diag(const Phys<T>& P, const T* macro, const T* phi_prev, double* partial, int nparts,
                        const int* err, double* out, cudaStream_t s) {
  cudaError_t e = launch_maybe_dependent(true, k_diag_partial<T>, dim3(nparts), dim3(DIAG_THREADS), 0, s, P, macro,
                                         phi_prev, partial);
  if (e == cudaSuccess)
    e = launch_maybe_dependent(true, k_diag_final<T>, dim3(1), dim3(DIAG_THREADS), 0, s, (const double*)partial, nparts,
                               err, out);
  return e;
}

template <typename T>
cudaError_t launch_obs_links(const Phys<T>& P, const unsigned char* solid, uint16_t* obs, cudaStream_t s) {
  k_obs_links<T><<<row_grid(P.nx, P.ny, OBS_THREADS), OBS_THREADS, 0, s>>>(P, solid, obs);
  return cudaGetLastError();
}

template <class C, int MODEL, int MODE, bool UR, bool MOM>
static cudaError_t obs_passes(const Phys<typename C::value_t>& P, const Bufs<typename C::value_t>& B,
                              typename C::value_t* phis, typename C::value_t* mus, cudaStream_t s) {
  using T = typename C::value_t;
  const dim3 grid = row_grid(P.nx, P.ny, OBS_THREADS);
  const int fill_blocks = (P.obs_nfill + OBS_THREADS - 1) / OBS_THREADS;
  k_obs_phi<C, MODE == MODE_INIT ? MODE_INIT : MODE_STEP><<<grid, OBS_THREADS, 0, s>>>(P, B, phis, 0, P.nx, 0);
  if (MODEL == MODEL_CH) {
    k_obs_mu<T><<<grid, OBS_THREADS, 0, s>>>(P, phis, mus, 0, P.nx, 0);
    if (fill_blocks) k_obs_fill<T><<<fill_blocks, OBS_THREADS, 0, s>>>(P, mus);
  }
  k_obs_node<C, MODEL, MODE, UR, MOM><<<grid, OBS_THREADS, 0, s>>>(P, B, phis, mus);
  return cudaGetLastError();
}

template <class C, int MODEL, bool MOM = sizeof(typename C::value_t) == 4>
static cudaError_t obs_model(int mode, const Phys<typename C::value_t>& P, const Bufs<typename C::value_t>& B,
                             typename C::value_t* phis, typename C::value_t* mus, bool unit_rates,
                             cudaStream_t s) {
  switch (mode) {
    case MODE_STEP:
      return unit_rates ? obs_passes<C, MODEL, MODE_STEP, true, MOM>(P, B, phis, mus, s)
                        : obs_passes<C, MODEL, MODE_STEP, false, MOM>(P, B, phis, mus, s);
    case MODE_MACRO: return obs_passes<C, MODEL, MODE_MACRO, false, MOM>(P, B, phis, mus, s);
    case MODE_HIST: return obs_passes<C, MODEL, MODE_HIST, false, MOM>(P, B, phis, mus, s);
    case MODE_INIT: return obs_passes<C, MODEL, MODE_INIT, false, MOM>(P, B, phis, mus, s);
    default: return cudaErrorInvalidValue;
  }
}

// 16-bit Allen-Cahn step with obstacles on the TMA kernel: phi and its fill over
// the region the blocks near obstacles read (P.obs_box; the whole grid
// without P.obs_near), then k_step_tma<..., OBS>, whose near blocks read phi
// from the plane and the others run the plain step's path.
template <class C>
static cudaError_t obs_step_tma(const Phys<typename C::value_t>& P, const Bufs<typename C::value_t>& B0,
                                typename C::value_t* phis, int* err, bool unit_rates, cudaStream_t s) {
  using T = typename C::value_t;
  const int x_lo = P.obs_near ? P.obs_box[0] : 0, x_hi = P.obs_near ? P.obs_box[1] : P.nx;
  const int y_lo = P.obs_near ? P.obs_box[2] : 0, y_hi = P.obs_near ? P.obs_box[3] : P.ny;
  const bool pass = x_hi > x_lo && y_hi > y_lo;
  if (pass)
    k_obs_phi<C, MODE_STEP><<<row_grid(x_hi - x_lo, y_hi - y_lo, OBS_THREADS), OBS_THREADS, 0, s>>>(P, B0, phis, x_lo,
                                                                                                   x_hi, y_lo);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  Bufs<T> B = B0;
  B.phis = phis;
  // the step is the phi pass's programmatic dependent only right after it
  return unit_rates ? launch_tma_variant<C, true, true>(P, B, err, s, pass)
                    : launch_tma_variant<C, false, true>(P, B, err, s, pass);
}

// Cahn-Hilliard step with obstacles on the TMA kernel: phi with its fill and
// mu_phi over the regions the blocks near obstacles read (P.obs_box,
// P.obs_box_mu; the whole grid without P.obs_near), the mu_phi fill, then
// k_step_tma_ch<..., OBS>, whose near blocks read both planes and the
// others run the plain step's path.
template <class C>
static cudaError_t obs_step_tma_ch(const Phys<typename C::value_t>& P0, const Bufs<typename C::value_t>& B0,
                                   typename C::value_t* phis, typename C::value_t* mus, int* err, bool unit_rates,
                                   cudaStream_t s) {
  using T = typename C::value_t;
  const bool nb = P0.obs_near != nullptr;
  const int* bp = P0.obs_box;
  const int* bm = P0.obs_box_mu;
  const int px0 = nb ? bp[0] : 0, px1 = nb ? bp[1] : P0.nx, py0 = nb ? bp[2] : 0, py1 = nb ? bp[3] : P0.ny;
  const int mx0 = nb ? bm[0] : 0, mx1 = nb ? bm[1] : P0.nx, my0 = nb ? bm[2] : 0, my1 = nb ? bm[3] : P0.ny;
  const int fill_blocks = (P0.obs_nfill + OBS_THREADS - 1) / OBS_THREADS;
  // phi pass (a plain launch: it reads the previous step's populations),
  // then the mu_phi pass, the fill and the step, each a programmatic
  // dependent of the kernel before it (each waits for that kernel's output)
  bool prev = false;  // a pass was launched just before
  cudaError_t e = cudaSuccess;
  if (px1 > px0 && py1 > py0) {
    k_obs_phi<C, MODE_STEP><<<row_grid(px1 - px0, py1 - py0, OBS_THREADS), OBS_THREADS, 0, s>>>(P0, B0, phis, px0,
                                                                                               px1, py0);
    e = cudaGetLastError();
    prev = true;
  }
  if (e == cudaSuccess && mx1 > mx0 && my1 > my0) {
    e = launch_maybe_dependent(prev, k_obs_mu<T>, row_grid(mx1 - mx0, my1 - my0, OBS_THREADS), dim3(OBS_THREADS), 0, s,
                               P0, (const T*)phis, mus, mx0, mx1, my0);
    prev = true;
  }
  if (e == cudaSuccess && fill_blocks) {
    e = launch_maybe_dependent(prev, k_obs_fill<T>, dim3(fill_blocks), dim3(OBS_THREADS), 0, s, P0, mus);
    prev = true;
  }
  if (e != cudaSuccess) return e;
  Bufs<T> B = B0;
  B.phis = phis;
  B.mus = mus;
  Phys<T> P = P0;
  P.seg_rows = tma_ch_segment_rows<C>(P.nx, P.ny);
  if (P.seg_rows == LY)
    return unit_rates ? launch_tma_ch_seg<C, true, false, true>(P, B, err, s, prev)
                      : launch_tma_ch_seg<C, false, false, true>(P, B, err, s, prev);
  return unit_rates ? launch_tma_ch_seg<C, true, true, true>(P, B, err, s, prev)
                    : launch_tma_ch_seg<C, false, true, true>(P, B, err, s, prev);
}

// Allen-Cahn with obstacles in the node update's form MOM.
template <class C, bool MOM>
static cudaError_t obs_ac(int mode, const Phys<typename C::value_t>& P, const Bufs<typename C::value_t>& B,
                          typename C::value_t* phis, typename C::value_t* mus, bool unit_rates, int* err, bool use_tma,
                          cudaStream_t s) {
  if (use_tma && mode == MODE_STEP && P.nx >= 4 * XPAD) {
    if constexpr (C::dev) return obs_step_tma<C>(P, B, phis, err, unit_rates, s);
    else if (P.obs_near && P.pitch <= TILE_MAX_PITCH)
      return unit_rates ? launch_tile_kernel<C, MODEL_AC, MODE_STEP, true, true, MOM>(P, B, s)
                        : launch_tile_kernel<C, MODEL_AC, MODE_STEP, false, true, MOM>(P, B, s);
  }
  return obs_model<C, MODEL_AC, MOM>(mode, P, B, phis, mus, unit_rates, s);
}

template <class C>
cudaError_t launch_obs(int model, int mode, const Phys<typename C::value_t>& P, const Bufs<typename C::value_t>& B,
                       typename C::value_t* phis, typename C::value_t* mus, bool unit_rates, bool moments, int* err,
                       bool use_tma, cudaStream_t s) {
  if (!P.obs || !phis || (model == MODEL_CH && !mus)) return cudaErrorInvalidValue;
  if (model == MODEL_CH) {
    if (use_tma && mode == MODE_STEP && P.nx >= 4 * XPAD)
      return obs_step_tma_ch<C>(P, B, phis, mus, err, unit_rates, s);
    return obs_model<C, MODEL_CH>(mode, P, B, phis, mus, unit_rates, s);
  }
  constexpr bool fp32 = sizeof(typename C::value_t) == 4;
  if constexpr (!fp32)
    if (moments) return obs_ac<C, true>(mode, P, B, phis, mus, unit_rates, err, use_tma, s);
  return obs_ac<C, fp32>(mode, P, B, phis, mus, unit_rates, err, use_tma, s);
}

// Blocks of an adjoint node pass (each leaves a pair of dJ/dG partial sums).
template <typename T>
long long adjoint_blocks(int nx, int ny) {
  const dim3 b = tile_shape<PopPlain<T>>(nx, ny, false);
  return std::max((long long)((nx + ADJ_THREADS - 1) / ADJ_THREADS) * ny,
                  (long long)((nx + b.x - 1) / b.x) * ((ny + b.y - 1) / b.y));
}

// One adjoint step (or, with hist_only, the adjoint of the history set-up at
// t = 0 without the reverse streaming).  state: snapshot of the step's input
// state (f* set, g* set of pop_bytes each, then the 5 history planes).  At unit
// rates the compact passes, each a programmatic dependent of the one before.
template <typename T>
cudaError_t launch_adjoint_step(const Phys<T>& P, const void* state, long long pop_bytes, const AdjBufs& A,
                                double* gacc, bool hist_only, bool unit_rates, cudaStream_t s) {
  unit_rates = unit_rates && P.pitch <= TILE_MAX_PITCH;
  const T* fin = static_cast<const T*>(state);
  const T* gin = reinterpret_cast<const T*>(static_cast<const unsigned char*>(state) + pop_bytes);
  const T* hist = reinterpret_cast<const T*>(static_cast<const unsigned char*>(state) + 2 * pop_bytes);
  T *phi = static_cast<T*>(A.phi), *lext = static_cast<T*>(A.lext), *lh = static_cast<T*>(A.lh);
  T *lf = static_cast<T*>(A.lf), *lg = static_cast<T*>(A.lg);
  T *lp9 = static_cast<T*>(A.lp9), *lfp = static_cast<T*>(A.lfp), *lgp = static_cast<T*>(A.lgp);
  const dim3 grid((P.nx + ADJ_THREADS - 1) / ADJ_THREADS, P.ny), block(ADJ_THREADS);
  const int ex = P.nx + 2 * P.wall_x, ey = P.ny + 2 * P.wall_y;
  const dim3 egrid((ex + ADJ_THREADS - 1) / ADJ_THREADS, ey);
  long long parts = (long long)grid.x * grid.y;
  cudaError_t e = cudaSuccess;
  if (unit_rates) {
    const dim3 b = tile_shape<PopPlain<T>>(P.nx, P.ny, false);
    const dim3 tiles((P.nx + b.x - 1) / b.x, (P.ny + b.y - 1) / b.y);
    parts = (long long)tiles.x * tiles.y;
    // (the node pass is a plain launch: the copies and kernels before it on the
    // stream may write the state or lambda)
    e = launch_maybe_dependent(false, k_adj_tile<T>, tiles, b, sizeof(T) * (b.x + 2) * (b.y + 2), s, P, fin, gin, hist,
                               phi, (const T*)lf, (const T*)lg, lh, lp9, lfp, lgp, A.gpart, hist_only ? 1 : 0);
    if (e == cudaSuccess) e = launch_maybe_dependent(true, k_adj_gather4<T>, egrid, block, 0, s, P, (const T*)lp9, lext);
  } else {
    k_adj_phi<T><<<grid, block, 0, s>>>(P, fin, phi);
    k_adj_node<T><<<grid, block, 0, s>>>(P, fin, gin, hist, phi, lf, lg, lh, lp9, lfp, lgp, A.gpart, hist_only ? 1 : 0);
    k_adj_gather<T><<<egrid, block, 0, s>>>(P, lp9, lext);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess && P.wall_y)
    e = launch_maybe_dependent(unit_rates, k_adj_fold_y<T>, dim3((ex + ADJ_THREADS - 1) / ADJ_THREADS), block, 0, s, P,
                               (const T*)phi, lext);
  if (e == cudaSuccess && P.wall_x)
    e = launch_maybe_dependent(unit_rates, k_adj_fold_x<T>, dim3((P.ny + ADJ_THREADS - 1) / ADJ_THREADS), block, 0, s,
                               P, (const T*)phi, lext);
  if (e == cudaSuccess && !hist_only) {
    if (unit_rates) {
      e = launch_maybe_dependent(true, k_adj_stream14<T>, grid, block, 0, s, P, (const T*)lfp, (const T*)lgp,
                                 (const T*)lext, lf, lg);
    } else {
      k_adj_stream<T><<<grid, block, 0, s>>>(P, lfp, lgp, lext, lf, lg);
      e = cudaGetLastError();
    }
  }
  if (e == cudaSuccess)
    e = launch_maybe_dependent(unit_rates, k_adj_reduce<T>, dim3(1), dim3(256), 0, s, (const double*)A.gpart, parts, gacc);
  return e;
}

template <typename T>
cudaError_t launch_adjoint_seed(const Phys<T>& P, const double* djdphi, const AdjBufs& A, cudaStream_t s) {
  const dim3 grid((P.nx + ADJ_THREADS - 1) / ADJ_THREADS, P.ny);
  k_adj_seed<T><<<grid, ADJ_THREADS, 0, s>>>(P, djdphi, static_cast<T*>(A.lf), static_cast<T*>(A.lg),
                                             static_cast<T*>(A.lh));
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_adjoint_init(const Phys<T>& P, const AdjBufs& A, double* out, cudaStream_t s) {
  const dim3 grid((P.nx + ADJ_THREADS - 1) / ADJ_THREADS, P.ny);
  k_adj_init<T><<<grid, ADJ_THREADS, 0, s>>>(P, static_cast<const T*>(A.lf), static_cast<const T*>(A.lext), out);
  return cudaGetLastError();
}

// the codec-typed wrappers of one storage codec
#define PFLBM_INSTANTIATE_CODEC(C)                                                                  \
  template cudaError_t launch_march<C>(int, int, const Phys<C::value_t>&, const Bufs<C::value_t>&,  \
                                       cudaStream_t);                                               \
  template cudaError_t launch_obs<C>(int, int, const Phys<C::value_t>&, const Bufs<C::value_t>&,    \
                                     C::value_t*, C::value_t*, bool, bool, int*, bool, cudaStream_t);     \
  template void obs_step_grid<C>(int, int, bool, int*, int*);

#define PFLBM_INSTANTIATE_DEV(C)                                                                    \
  PFLBM_INSTANTIATE_CODEC(C)                                                                        \
  template cudaError_t launch_step_tma<C>(const Phys<C::value_t>&, const Bufs<C::value_t>&, int*,   \
                                          bool, cudaStream_t);                                      \
  template cudaError_t launch_step_tma_ch<C>(const Phys<C::value_t>&, const Bufs<C::value_t>&, int*, \
                                             bool, cudaStream_t);                                   \
  template cudaError_t launch_pull_export<C>(const Phys<C::value_t>&, const void*, int, int, double*, \
                                             double, int, int, int, int, cudaStream_t);             \
  template cudaError_t launch_restream<C>(const Phys<C::value_t>&, const C::value_t*, void*, int,   \
                                          cudaStream_t);

// the arithmetic-type wrappers
#define PFLBM_INSTANTIATE(T)                                                                        \
  PFLBM_INSTANTIATE_CODEC(PopPlain<T>)                                                              \
  template cudaError_t launch_tile<PopPlain<T>>(int, int, const Phys<T>&, const Bufs<T>&, bool, bool, \
                                                cudaStream_t);                                     \
  template cudaError_t launch_pull<T>(const Phys<T>&, const T*, T*, cudaStream_t);                \
  template cudaError_t launch_unstream<T>(const Phys<T>&, const T*, T*, cudaStream_t);            \
  template cudaError_t launch_export<T>(const Phys<T>&, const T*, int, int, double*, double, int,  \
                                        int, int, int, cudaStream_t);                              \
  template cudaError_t launch_import<T>(const Phys<T>&, const double*, T*, int, int, double,      \
                                        cudaStream_t);                                             \
  template cudaError_t launch_diag<T>(const Phys<T>&, const T*, const T*, double*, int, const int*, \
                                      double*, cudaStream_t);                                      \
  template cudaError_t launch_adjoint_step<T>(const Phys<T>&, const void*, long long, const AdjBufs&, \
                                              double*, bool, bool, cudaStream_t);                 \
  template long long adjoint_blocks<T>(int, int);                                                   \
  template cudaError_t launch_adjoint_seed<T>(const Phys<T>&, const double*, const AdjBufs&,      \
                                              cudaStream_t);                                      \
  template cudaError_t launch_adjoint_init<T>(const Phys<T>&, const AdjBufs&, double*, cudaStream_t); \
  template cudaError_t launch_obs_links<T>(const Phys<T>&, const unsigned char*, uint16_t*, cudaStream_t);

}  // namespace pflbm
