// steps_1d.cuh -- whole time steps of a short one-dimensional problem (FP64) in
// one launch of one block.
//
// A tube of a few hundred cells fills a few warps; the 13 kernels of the
// general step spend their time on launches and on finding their data in L2.
// One block needs __syncthreads between the phases instead of kernel boundaries
// and finds what the phase before wrote in its own L1, and a run needs no launch
// a step.  Its FP64 pipes are one SM's, so the general step is the faster one
// above kMaxCells1D cells: a step of the R = 2 shock tube takes, in one block
// and in general, 81 and 124 us at 128 cells, 114 and 142 at 256, 153 and 152 at
// 512, 168 and 155 at 640 (R = 1 and 3 cross between 512 and 640 too).
#pragma once

#include "gpmood_kernels.cuh"

namespace gpm {

// the states of all faces of the row, formed by one lane a cell and variable:
// st[east, west][variable][cell + 1], cells -1 .. nx.  The same sums as the
// first-pass face kernel forms of the embedded 1D weights, whose off-row
// coefficients are zero.
template <int R>
__device__ __forceinline__ void states_1d(const double* X, const Grid& g,
                                          const ParityW<double>& W, double* st) {
  const int n = g.nx + 2;
  for (int t = threadIdx.x; t < 4 * n; t += blockDim.x) {
    const int v = t / n, c = t - v * n;
    const double* x0 = X + gidx(g, v, c - 1, 0);
    double east, west;
    if constexpr (R == 0) {
      east = west = *x0;
    } else {
      double x[2 * R + 1];
#pragma unroll
      for (int a = -R; a <= R; ++a) x[a + R] = x0[a];
      uint32_t top = (uint32_t)FXD_EMIN << 20;
#pragma unroll
      for (int a = 0; a <= 2 * R; ++a) top = max(top, fxd_hi(x[a]) & 0x7fffffffu);
      const int E = (int)(top >> 20);
      const uint32_t special = E == 0x7ff ? 0x7ff80000u : 0u;
      fxd_acc even = {0, 0, 0}, odd = {0, 0, 0};
      const long long m = fxd_from_double(x[R], E);
      fxd_mac(&even, W.cx[0][0].x, W.cx[0][0].y, fxd_limb_hi(m), fxd_limb_lo(m));
#pragma unroll
      for (int a = 1; a <= R; ++a) {
        const long long p = fxd_from_double(x[R + a], E), q = fxd_from_double(x[R - a], E);
        const int2 ce = W.cx[0][2 * a - 1], co = W.cx[0][2 * a];
        fxd_mac(&even, ce.x, ce.y, fxd_limb_hi(p + q), fxd_limb_lo(p + q));
        fxd_mac(&odd, co.x, co.y, fxd_limb_hi(p - q), fxd_limb_lo(p - q));
      }
      const long long e = fxd_round(even), o = fxd_round(odd);
      east = fxd_to_double(e + o, E, W.off, special);
      west = fxd_to_double(e - o, E, W.off, special);
    }
    st[v * n + c] = east;
    st[(4 + v) * n + c] = west;
  }
}

// the fluxes of all faces from the states, one lane a face
template <int R>
__device__ __forceinline__ void fluxes_1d(const StageArgs<double>& A, const Grid& g,
                                          const ParityW<double>& W, const double* st) {
  const int n = g.nx + 2;
  for (int f = threadIdx.x; f <= g.nx; f += blockDim.x) {
    double a[4], b[4], h[4], pl, pr;
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      a[v] = st[v * n + f];            // east state of cell f - 1
      b[v] = st[(4 + v) * n + f + 1];  // west state of cell f
    }
    riemann_x<double>(g.riemann, a, b, g.gamma, h, pl, pr);
    // the two equal points of weight 1/2 (R = 0: one point)
#pragma unroll
    for (int v = 0; v < 4; ++v)
      A.Fx[fxidx(g, v, f, 0)] = fma(W.w[0], R == 0 ? h[v] : add_rn(h[v], h[v]), 0.0);
    A.fbx[f] = (uint8_t)((pos_finite(a[0]) && pos_finite(pl) ? 0 : 1) |
                         (pos_finite(b[0]) && pos_finite(pr) ? 0 : 2));
  }
}

template <int R>
__global__ void __launch_bounds__(256) k_steps_1d(const __grid_constant__ Steps1D S,
                                                  const __grid_constant__ Grid g,
                                                  const __grid_constant__ Detect D,
                                                  const __grid_constant__ ParityW<double> W,
                                                  const __grid_constant__ DirectW<double> Wd,
                                                  const __grid_constant__ Cascade C) {
  extern __shared__ __align__(16) double st1d[];
  __shared__ double warp_rate[8];
  __shared__ int go, bad_rate, queued;
  __shared__ StageC coef;
  Scalars* sc = S.sc;
  const int tid = threadIdx.x, nbuf = S.sch.nbuf;
  if (tid == 0) sc->launches += 1;
  int rot = S.rot;
  for (int step = 0; step < S.nsteps; ++step, rot = (rot + S.sch.advance) % nbuf) {
    // the gate of queued steps (k_step_gate)
    if (tid == 0) {
      const Control c = sc->ctl;
      go = sc->err == 0 && !(c.clip && !(sc->t < c.t_end * (1.0 - 1e-14)));
      bad_rate = 0;
      queued = 0;
    }
    __syncthreads();
    if (!go) return;
    // the time step (k_dt_reduce, k_dt_finalize)
    const double* U0 = S.U[rot];
    double best = 0.0;
    bool bad = false;
    if (!(sc->ctl.fixed_dt > 0.0))
      for (int i = tid; i < g.nx; i += blockDim.x) {
        double a;
        if (!cell_rate_at(U0, nullptr, g, i, 0, a)) bad = true;
        else best = max_num(a, best);
      }
    for (int o = 16; o > 0; o >>= 1)
      best = max_num(__shfl_xor_sync(0xffffffffu, best, o), best);
    if ((tid & 31) == 0) warp_rate[tid >> 5] = best;
    if (bad) bad_rate = 1;
    __syncthreads();
    if (tid == 0) {
      const Control c = sc->ctl;
      double r = g.rate_floor, dt;
      for (int w = 0; w < 8; ++w) r = max_num(warp_rate[w], r);
      if (c.fixed_dt > 0.0) {
        dt = c.fixed_dt;
      } else {
        dt = c.cfl / r;
        if (c.clip && sc->t + dt > c.t_end) dt = c.t_end - sc->t;
      }
      if (bad_rate || !(dt > 0.0) || !isfinite(dt)) sc->err |= kErrDt;
      sc->dt = dt;
      sc->rate_bits = 0ull;
      sc->rate_ready = 0;
      sc->rate_bad = 0;
      for (int s = 0; s < 5; ++s) sc->iters[s] = sc->nbad_first[s] = sc->nbad_total[s] = sc->nfog_pad[s] = 0;
    }
    __syncthreads();
    const double t0 = sc->t, dt = sc->dt;
    for (int s = 0; s < S.sch.nstages; ++s) {
      const StageSpec p = S.sch.st[s];
      StageArgs<double> A;
      double* X = S.U[(rot + p.in) % nbuf];
      A.X = A.Xr = X;
      A.U0 = S.U[(rot + p.u0) % nbuf];
      A.out = S.U[(rot + p.out) % nbuf];
      A.outr = nullptr;
      A.W = p.w >= 0 ? S.U[(rot + p.w) % nbuf] : nullptr;
      A.out2 = p.out2 >= 0 ? S.U[(rot + p.out2) % nbuf] : nullptr;
      A.h = p.h;
      A.ca = p.ca;
      A.cb = p.cb;
      A.wa = p.wa;
      A.wb = p.wb;
      A.Fx = S.Fx;
      A.Fy = S.Fy;
      A.fbx = S.fb;
      A.fby = S.fb + (size_t)(g.nx + 1) * g.ny;
      A.ord = S.ord + (size_t)s * g.nx;
      A.first = S.first + (size_t)s * g.nx;
      A.queue = S.queue[0];
      A.qcount = &queued;
      A.sc = sc;
      A.scw = sc;
      A.stage = s;
      const long long ng = ghost_count(g);
      for (long long k = tid; k < ng; k += blockDim.x) fill_ghost(X, nullptr, g, t0 + p.tfrac * dt, k);
      if (tid == 0) coef = stage_coeffs<double>(A, g, dt);
      __syncthreads();
      states_1d<R>(X, g, W, st1d);
      __syncthreads();
      fluxes_1d<R>(A, g, W, st1d);
      __syncthreads();
      for (int i = tid & ~31; i < g.nx; i += blockDim.x)
        update_cell_w<double>(A, g, D, Wd, Wd.d2x, Wd.d2y, i + (tid & 31), 0, 0, coef);
      __syncthreads();
      MoodArgs M;
      M.queue[0] = S.queue[0];
      M.queue[1] = S.queue[1];
      M.stamp = S.stamp;
      M.stamp_stride = g.nx;
      M.count = &queued;
      M.sc = sc;
      const SingleSite<double> site{A, g, D, Wd.d2x, Wd.d2y, &coef};
      mood_loop_body<double>(site, M, Wd, C, s, false);
      __syncthreads();
    }
    // the end of the step (k_finish_step)
    if (tid == 0 && sc->err == 0) {
      sc->t = t0 + dt;
      sc->nsteps += 1;
    }
    __syncthreads();
  }
}

}  // namespace gpm
