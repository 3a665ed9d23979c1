// kernels_impl.cuh -- launcher bodies, instantiated once per precision.
#pragma once

#include <type_traits>

#include "adjoint_kernels.cuh"
#include "faces_fp64.cuh"
#include "gpmood_kernels.cuh"
#include "gpmood_launch.h"
#include "steps_1d.cuh"

namespace gpm {

// calls f(std::integral_constant<int, R>) for the top radius
template <class F>
static cudaError_t with_radius(int top, F&& f) {
  switch (top) {
    case 0: return f(std::integral_constant<int, 0>());
    case 1: return f(std::integral_constant<int, 1>());
    case 2: return f(std::integral_constant<int, 2>());
    default: return f(std::integral_constant<int, 3>());
  }
}

// FP64 faces of the directions in dirs (1 x, 2 y, 3 both)
template <class Real>  // double; a template, so that only its own files instantiate the kernels
static cudaError_t faces_fx(int top, int dirs, const StageArgs<Real>& A, const Grid& g,
                            const ParityW<Real>& W, cudaStream_t st) {
  const int nseg = fx_segments(g.nx), nb = fx_bands(1, &g.nx, &g.ny);
  const int units = nseg * fx_chunks(g.ny, nb);
  return with_radius(top, [&](auto r) {
    constexpr int R = decltype(r)::value;
    return launch_ks(k_faces_fx<R>, dim3(fx_grid(units)), dim3(kFxThreads), sizeof(FxShared<R>),
                     st, A, g, W, nseg, nb, units, dirs);
  });
}

template <int R>
static cudaError_t faces_r(int dir, const StageArgs<float>& A, const Grid& g,
                           const ParityW<float>& W, cudaStream_t st) {
  dim3 blk(32, kFaceWarps);
  if (dir == 0) {
    dim3 gx((g.nx + 1 + kSegFaces - 1) / kSegFaces, (g.ny + kFaceWarps - 1) / kFaceWarps);
    return launch_k(k_faces<R, float, 0, kFaceWarps>, gx, blk, st, A, g, W);
  }
  dim3 gy((g.nx + kFaceWarps - 1) / kFaceWarps, (g.ny + 1 + kSegFaces - 1) / kSegFaces);
  return launch_k(k_faces<R, float, 1, kFaceWarps>, gy, blk, st, A, g, W);
}

template <class Real>
cudaError_t Launch<Real>::faces(int top, int dir, const StageArgs<Real>& A, const Grid& g,
                                const ParityW<Real>& W, cudaStream_t st) {
  if constexpr (sizeof(Real) == sizeof(double)) return faces_fx(top, 1 << dir, A, g, W, st);
  else return with_radius(top, [&](auto r) { return faces_r<decltype(r)::value>(dir, A, g, W, st); });
}

template <class Real>
cudaError_t Launch<Real>::faces_xy(int top, const StageArgs<Real>& A, const Grid& g,
                                   const ParityW<Real>& W, cudaStream_t st) {
  if constexpr (sizeof(Real) == sizeof(double)) {
    return faces_fx(top, 3, A, g, W, st);
  } else {
    return with_radius(top, [&](auto r) {
      constexpr int R = decltype(r)::value;
      dim3 grd((g.nx + 1 + kSegFaces - 1) / kSegFaces, (g.ny + 1 + kXYBand - 1) / kXYBand);
      return launch_ks(k_faces_xy<R, Real>, grd, dim3(32, kXYRows), sizeof(XYShared<R, Real>),
                       st, A, g, W);
    });
  }
}

// the shared-memory limit of a face kernel of either precision
template <class Kernel>
static cudaError_t shared_limit(Kernel k, size_t bytes) {
  return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}
template <class Real, class F>
static cudaError_t every_radius(F&& f) {
  cudaError_t e = cudaSuccess;
  for (int r = 0; r <= 3 && e == cudaSuccess; ++r) e = with_radius(r, f);
  return e;
}

template <class Real>
cudaError_t Launch<Real>::steps_1d(int top, const Steps1D& S, const Grid& g, const Detect& D,
                                   const ParityW<Real>& W, const DirectW<Real>& Wd,
                                   const Cascade& C, cudaStream_t st) {
  if constexpr (sizeof(Real) == sizeof(double))
    return with_radius(top, [&](auto r) {
      constexpr int R = decltype(r)::value;
      return launch_ks(k_steps_1d<R>, dim3(1), dim3(256), 8 * sizeof(double) * (g.nx + 2), st, S, g,
                       D, W, Wd, C);
    });
  else return cudaErrorInvalidValue;
}

template <class Real>
cudaError_t Launch<Real>::prepare() {
  return every_radius<Real>([](auto r) {
    constexpr int R = decltype(r)::value;
    if constexpr (sizeof(Real) == sizeof(double)) {
      cudaError_t e = shared_limit(k_faces_fx<R>, sizeof(FxShared<R>));
      return e != cudaSuccess ? e : shared_limit(k_steps_1d<R>, 8 * sizeof(double) * (kMaxCells1D + 2));
    } else {
      return shared_limit(k_faces_xy<R, Real>, sizeof(XYShared<R, Real>));
    }
  });
}

template <class Real>
cudaError_t Launch<Real>::update_first(const StageArgs<Real>& A, const Grid& g, const Detect& D,
                                       const DirectW<Real>& Wd, cudaStream_t st) {
  dim3 blk(32, 8);
  dim3 grd((g.nx + 31) / 32, (g.ny + 7) / 8);
  return launch_k(k_update_first<Real>, grd, blk, st, A, g, D, Wd);
}

template <class Real>
cudaError_t Launch<Real>::mood_loop(const StageArgs<Real>& A, const MoodArgs& M, const Grid& g,
                                    const Detect& D, const DirectW<Real>& Wd, const Cascade& C,
                                    int stage, const LoopTail& T, int blocks, int coop,
                                    cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(256);
  cfg.stream = st;
  // cooperative: the launch fails rather than run a grid whose blocks cannot
  // all be resident at once (the barriers need them all)
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = coop ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, k_mood_loop<Real>, A, M, g, D, Wd, C, stage, T);
}

template <class Real>
int Launch<Real>::mood_loop_blocks() {
  int dev = 0, sms = 0, occ = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_mood_loop<Real>, 256, 0) !=
          cudaSuccess || sms <= 0 || occ <= 0) {
    cudaGetLastError();
    return 0;
  }
  // two blocks an SM where they fit: enough warps to hide the FP64 latency
  // of the few cells an iteration works on, few arrivals per barrier
  return sms * (occ < 2 ? occ : 2);
}

template <int R, int FW>
static void faces_batch_r(int dir, const StageArgs<float>& B, const Prob* probs,
                          const Scalars* psc, const Item* items, int nitems,
                          const ParityW<float>& W, cudaStream_t st) {
  dim3 blk(32, FW);  // one block per item
  if (dir == 0) k_faces_batch<R, float, 0, FW><<<nitems, blk, 0, st>>>(B, probs, psc, items, W);
  else k_faces_batch<R, float, 1, FW><<<nitems, blk, 0, st>>>(B, probs, psc, items, W);
}

template <class Real>
cudaError_t LaunchB<Real>::faces(int top, int dir, int fw, const StageArgs<Real>& B,
                                 const Prob* probs, const Scalars* psc, const Item* items,
                                 int nitems, const ParityW<Real>& W, cudaStream_t st) {
  if (nitems <= 0) return cudaSuccess;
  if constexpr (sizeof(Real) == sizeof(double)) return cudaErrorInvalidValue;  // FP64: faces_xy
  else return with_radius(top, [&](auto r) {
    constexpr int R = decltype(r)::value;
    if (fw == 4) faces_batch_r<R, 4>(dir, B, probs, psc, items, nitems, W, st);
    else faces_batch_r<R, 8>(dir, B, probs, psc, items, nitems, W, st);
    return cudaGetLastError();
  });
}

template <class Real>
cudaError_t LaunchB<Real>::faces_xy(int top, const StageArgs<Real>& B, const Prob* probs,
                                    const Scalars* psc, const Item* items, int nitems,
                                    const ParityW<Real>& W, cudaStream_t st) {
  if (nitems <= 0) return cudaSuccess;
  return with_radius(top, [&](auto r) {
    constexpr int R = decltype(r)::value;
    if constexpr (sizeof(Real) == sizeof(double))
      return launch_ks(k_faces_fx_batch<R>, dim3(fx_grid(nitems)), dim3(kFxThreads),
                       sizeof(FxShared<R>), st, B, probs, psc, items, nitems, W);
    else
      return launch_ks(k_faces_xy_batch<R, Real>, dim3(nitems), dim3(32, kXYRows),
                       sizeof(XYShared<R, Real>), st, B, probs, psc, items, W);
  });
}

template <class Real>
cudaError_t LaunchB<Real>::prepare() {
  return every_radius<Real>([](auto r) {
    constexpr int R = decltype(r)::value;
    if constexpr (sizeof(Real) == sizeof(double))
      return shared_limit(k_faces_fx_batch<R>, sizeof(FxShared<R>));
    else return shared_limit(k_faces_xy_batch<R, Real>, sizeof(XYShared<R, Real>));
  });
}

template <class Real>
cudaError_t LaunchB<Real>::update(const StageArgs<Real>& B, const Prob* probs, const Scalars* psc,
                                  const Item* items, int nitems, int blocks,
                                  const DirectW<Real>& Wd, cudaStream_t st) {
  if (nitems <= 0) return cudaSuccess;
  k_update_batch<Real><<<blocks, dim3(32, 8), 0, st>>>(B, probs, psc, items, nitems, Wd);
  return cudaGetLastError();
}

template <class Real>
cudaError_t LaunchB<Real>::mood_loop(const StageArgs<Real>& B, const MoodArgs& M,
                                     const Prob* probs, const Scalars* psc, int nprob,
                                     const DirectW<Real>& Wd, const Cascade& C, int stage,
                                     int blocks, int coop, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(256);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = coop ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, k_mood_loop_batch<Real>, B, M, probs, psc, nprob, Wd, C, stage);
}

template <class Real>
int LaunchB<Real>::mood_loop_blocks() {
  int dev = 0, sms = 0, occ = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_mood_loop_batch<Real>, 256, 0) !=
          cudaSuccess || sms <= 0 || occ <= 0) {
    cudaGetLastError();
    return 0;
  }
  return sms * (occ < 2 ? occ : 2);
}

template <class Real>
cudaError_t LaunchA<Real>::frozen_stage(const StageArgs<Real>& A, const Grid& g,
                                        const DirectW<Real>& Wd, cudaStream_t st) {
  const long long nfx = (long long)(g.nx + 1) * g.ny, nfy = (long long)g.nx * (g.ny + 1);
  k_faces_frozen<Real, 0><<<(int)((nfx + 127) / 128), 128, 0, st>>>(A, g, Wd);
  k_faces_frozen<Real, 1><<<(int)((nfy + 127) / 128), 128, 0, st>>>(A, g, Wd);
  k_update_frozen<Real><<<dim3((g.nx + 31) / 32, (g.ny + 7) / 8), dim3(32, 8), 0, st>>>(A, g);
  return cudaGetLastError();
}

template <int R, class Real>
static cudaError_t adj_faces_r(const Real* X, const double* v, const uint8_t* ord,
                               const Grid& g, const ParityW<Real>& W, const DirectW<Real>& Wd,
                               const AdjFaces& Ax, const AdjFaces& Ay, cudaStream_t st) {
  // 4 warps a block: the reverse sweep holds ~150-250 registers a thread
  constexpr int FW = 4;
  dim3 blk(32, FW);
  dim3 gx((g.nx + 1 + kSegFaces - 1) / kSegFaces, (g.ny + FW - 1) / FW);
  k_adj_faces_sweep<R, Real, 0, FW><<<gx, blk, 0, st>>>(X, v, ord, g, W, Wd, Ax);
  dim3 gy((g.nx + FW - 1) / FW, (g.ny + 1 + kSegFaces - 1) / kSegFaces);
  k_adj_faces_sweep<R, Real, 1, FW><<<gy, blk, 0, st>>>(X, v, ord, g, W, Wd, Ay);
  return cudaGetLastError();
}

template <class Real>
cudaError_t LaunchA<Real>::adj_faces(const double* X, void* Xr, const double* v,
                                     const uint8_t* ord, const Grid& g, const ParityW<Real>& W,
                                     const DirectW<Real>& Wd, const AdjFaces& Ax,
                                     const AdjFaces& Ay, cudaStream_t st) {
  const Real* XR;
  if (sizeof(Real) == sizeof(double)) {
    XR = (const Real*)X;
  } else {
    k_to_real<Real><<<152 * 8, 256, 0, st>>>(X, (Real*)Xr, 4 * g.vstride);
    XR = (const Real*)Xr;
  }
  switch (Wd.top) {
    case 0: return adj_faces_r<0, Real>(XR, v, ord, g, W, Wd, Ax, Ay, st);
    case 1: return adj_faces_r<1, Real>(XR, v, ord, g, W, Wd, Ax, Ay, st);
    case 2: return adj_faces_r<2, Real>(XR, v, ord, g, W, Wd, Ax, Ay, st);
    default: return adj_faces_r<3, Real>(XR, v, ord, g, W, Wd, Ax, Ay, st);
  }
}

template <class Real>
cudaError_t LaunchA<Real>::adj_faces_stored(const void* st, const double* v, const uint8_t* ord,
                                            const Grid& g, const ParityW<Real>& W,
                                            const DirectW<Real>& Wd, const AdjFaces& Ax,
                                            const AdjFaces& Ay, cudaStream_t s) {
  const int qt = rule_q(Wd.top);
  const Real* t = (const Real*)st;
  const Real* xL = t;
  const Real* xR = t + 4LL * qt * Ax.nf;
  const Real* yL = t + 8LL * qt * Ax.nf;
  const Real* yR = yL + 4LL * qt * Ay.nf;
  k_adj_faces_stored<Real, 0><<<(int)((Ax.nf + 127) / 128), 128, 0, s>>>(xL, xR, qt, v, ord, g,
                                                                         W, Wd, Ax);
  k_adj_faces_stored<Real, 1><<<(int)((Ay.nf + 127) / 128), 128, 0, s>>>(yL, yR, qt, v, ord, g,
                                                                         W, Wd, Ay);
  return cudaGetLastError();
}

template <class Real>
cudaError_t LaunchA<Real>::adj_gather(const Grid& g, const GatherW<Real>& Wd, const AdjFaces& Ax,
                                      const AdjFaces& Ay, double* G, cudaStream_t st) {
  if constexpr (sizeof(Real) == sizeof(double)) {
    return with_radius(Wd.top, [&](auto r) {
      constexpr int R = decltype(r)::value;
      cudaError_t e = shared_limit(k_adj_gather_fx<R>, sizeof(GatherShared<R>));
      if (e != cudaSuccess) return e;
      dim3 grd((g.nx + 2 * g.H + 31) / 32, (g.ny + 2 * g.H + 7) / 8);
      k_adj_gather_fx<R><<<grd, 256, sizeof(GatherShared<R>), st>>>(g, Wd, Ax, Ay, G);
      return cudaGetLastError();
    });
  } else {
    const long long n = (long long)(g.nx + 2 * g.H) * (g.ny + 2 * g.H);
    k_adj_gather<Real><<<(int)((n + 255) / 256), 256, 0, st>>>(g, Wd, Ax, Ay, G);
    return cudaGetLastError();
  }
}

}  // namespace gpm
