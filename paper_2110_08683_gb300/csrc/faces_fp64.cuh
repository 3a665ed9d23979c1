// faces_fp64.cuh -- first-pass faces at the top radius, FP64.
//
// What bounds it: the FP64 pipe (64 cycles a warp instruction a
// sub-partition) in the Riemann solver, the integer pipes in the
// reconstruction (fixed_dot.h), which different warps of a block do side by
// side.  4096 x 1024 double Mach
// reflection, R = 3: 3.27 ms a launch, the FP64 pipe's share of it 2.4 ms (180
// instructions a face).  It was 11.1 ms with everything on the FP64 pipe (716
// instructions a face), 6.0 ms with the reconstruction's 396 taken off it,
// 4.6 ms with 180 for the solver's 320, and the rest is the split of the
// warps.
#pragma once

#include "gpmood_kernels.cuh"

namespace gpm {

// A block walks up segments of 32 cell columns in bands of 4 rows, with 8
// warps that reconstruct and 8 that solve.  Reconstructing warps w and w + 4
// form the states of the cells of row w on all four faces, two variables each
// (lane l holds cell (i0 + l, j0 + w), i0 = 31 seg - 1), into one of two shared
// buffers while the solving warps work on the other: one warp a row for the x
// faces, one for the y faces below the row.  Integer and FP64 work then run side by side;
// in a block whose warps all do the one and then the other they hardly
// overlapped (all blocks of an SM drift into step).  A row's warps sit on one
// sub-partition each, so the FP64 work is even.  The upper states of a band's
// last row wait in a third buffer for the band above.  Only the first band of
// a unit has a row (its lowest) that merely supplies states.
constexpr int kFxRows = 4;
constexpr int kFxThreads = 32 * 4 * kFxRows;

template <int R>
struct FxShared {
  static constexpr int Q = rule_q(R);
  struct Band {
    double x[2][Q][4][kFxRows][32];  // [east, west][point][variable][row][lane]
    double n[Q][4][kFxRows - 1][32]; // north states of rows 0-2
    double s[Q][4][kFxRows][32];     // south
  } band[2];
  double top[3][Q][4][32];           // north states of row 3, by band modulo 3
};

// barrier `id` among all threads of the block: wait, or only arrive
__device__ __forceinline__ void bar_wait(int id) {
  __syncwarp();
  asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(kFxThreads) : "memory");
}
__device__ __forceinline__ void bar_arrive(int id) {
  __threadfence_block();
  __syncwarp();
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "n"(kFxThreads) : "memory");
}
// barriers: buffer b is full 1 + b, empty 3 + b (0 is __syncthreads)

// the face states of one cell and variable along one axis, from its parity
// sums: point q of the plus side (east / north) goes to p[q * ps], of the
// minus side (west / south) to m[q * ms]
template <int R, int AXIS>
__device__ __forceinline__ void fx_states(const ReconFixed<R>& rc, const ParityW<double>& W,
                                          int npair, double* p, int ps, double* m, int ms) {
  constexpr int Q = rule_q(R);
  constexpr int NS = (Q + 1) / 2;
#pragma unroll
  for (int kk = 0; kk < NS; ++kk) {
    if (kk >= npair) break;
    long long T[2][2];
    rc.dot(AXIS == 0 ? W.cx[kk] : W.cy[kk], T);
    // even and odd along the axis: T[0][.] and T[1][.] for x, T[.][0] and T[.][1] for y
    const long long t01 = AXIS == 0 ? T[0][1] : T[1][0], t10 = AXIS == 0 ? T[1][0] : T[0][1];
    if ((Q & 1) && kk == Q / 2) {
      p[kk * ps] = rc.out(T[0][0] + t10, W);
      m[kk * ms] = rc.out(T[0][0] - t10, W);
    } else {
      const long long e = T[0][0] + t01, o = t10 + T[1][1];
      const long long e2 = T[0][0] - t01, o2 = t10 - T[1][1];
      p[kk * ps] = rc.out(e + o, W);
      m[kk * ms] = rc.out(e - o, W);
      p[(Q - 1 - kk) * ps] = rc.out(e2 + o2, W);
      m[(Q - 1 - kk) * ms] = rc.out(e2 - o2, W);
    }
  }
}

// a unit of work: segment seg, rows r0 .. r0 + 4 nb - 2 of faces (x faces of
// rows below ny, y faces up to ny).  Its bands: row j0 = r0 - 1 + 4 b on.
__device__ __forceinline__ int unit_bands(const Grid& g, int r0, int nb) {
  const int rows = g.ny + 2 - r0;  // of states, from r0 - 1 to ny
  const int need = (rows + kFxRows - 1) / kFxRows;
  return need < nb ? need : nb;
}

// the states of band rows j0 .. j0 + 3 of a segment: one reconstructing warp's
template <int R>
__device__ __forceinline__ void fx_produce(const double* X0, const Grid& g,
                                           const ParityW<double>& W, int seg, int j0, bool first,
                                           int dirs, typename FxShared<R>::Band& B,
                                           double (*top)[4][32]) {
  constexpr int Q = rule_q(R);
  constexpr int NS = (Q + 1) / 2;
  constexpr int kVar = kFxRows * 32, kVarN = (kFxRows - 1) * 32;
  const int lane = threadIdx.x & 31, row = (threadIdx.x >> 5) & 3;
  const int v0 = threadIdx.x >> 7 << 1;  // this warp's first variable
  const int i = seg * kSegFaces - 1 + lane, ic = i < g.nx ? i : g.nx, j = j0 + row;
  const bool xrow = (dirs & 1) && (!first || row > 0) && j < g.ny;
  const bool ystate = (dirs & 2) && j <= g.ny;
  if (!xrow && !ystate) return;
  // the 1D method's points all carry the same state: one pair is formed
  const int npair = g.dim == 1 ? 1 : NS;
  const double* X = X0 + v0 * g.vstride + (long long)(j + g.H) * g.pitch + (ic + g.H);
  const int pitch = g.pitch;
  double* xe = &B.x[0][0][v0][row][lane];
  double* xw = &B.x[1][0][v0][row][lane];
  double* ys = &B.s[0][v0][row][lane];
  const bool last = row == kFxRows - 1;
  double* yn = last ? &top[0][v0][lane] : &B.n[0][v0][row < kFxRows - 1 ? row : 0][lane];
  const int nv = last ? 32 : kVarN;  // stride of a variable
#pragma unroll 1
  for (int v = 0; v < 2; ++v, X += g.vstride, xe += kVar, xw += kVar, ys += kVar, yn += nv) {
    if constexpr (R == 0) {
      *xe = *xw = *yn = *ys = __ldg(X);
    } else {
      ReconFixed<R> rc;
      rc.sums([&](int a, int c) -> double { return __ldg(X + (long long)c * pitch + a); }, true);
      if (xrow) fx_states<R, 0>(rc, W, npair, xe, 4 * kVar, xw, 4 * kVar);
      if (ystate) fx_states<R, 1>(rc, W, npair, yn, 4 * nv, ys, 4 * kVar);
    }
  }
}

// the faces of one direction D of a row of the band: one solving warp.
// below: the upper states of the band below's last row.
template <int R, bool HLL>
__device__ __forceinline__ void fx_solve(const StageArgs<double>& A, const Grid& g,
                                         const ParityW<double>& W, int seg, int j0, bool first,
                                         int row, int d, const typename FxShared<R>::Band& B,
                                         const double (*below)[4][32]) {
  constexpr int Q = rule_q(R);
  constexpr int NS = (Q + 1) / 2;
  constexpr int kVar = kFxRows * 32, kVarN = (kFxRows - 1) * 32;
  const int lane = threadIdx.x & 31;
  const int i = seg * kSegFaces - 1 + lane, j = j0 + row;
  if (first && row == 0) return;  // the row is the unit below's
  // x face between (i-1, j) and (i, j); y face between (i, j-1) and (i, j)
  if (lane == 0 || (d == 0 ? (j >= g.ny || i > g.nx) : (j > g.ny || i >= g.nx))) return;
  const double* L = d == 0 ? &B.x[0][0][0][row][lane - 1]
                           : row == 0 ? &below[0][0][lane] : &B.n[0][0][row - 1][lane];
  const double* M = d == 0 ? &B.x[1][0][0][row][lane] : &B.s[0][0][row][lane];
  const int lv = d == 0 ? kVar : row == 0 ? 32 : kVarN;  // variable strides; points four apart
  const int mn = 1 + d, mt = 2 - d;                      // normal and tangential momentum
  const bool one = g.dim == 1;
  double F[4] = {0, 0, 0, 0};  // mass, normal, tangential, energy
  bool badL = false, badR = false;
  auto point = [&](int q, double* f) {
    const double* l = L + q * 4 * lv;
    const double* m = M + q * 4 * kVar;
    const double a[4] = {l[0], l[mn * lv], l[mt * lv], l[3 * lv]};
    const double c[4] = {m[0], m[mn * kVar], m[mt * kVar], m[3 * kVar]};
    double pl, pr;
    if (HLL) hll_x_fp64(a, c, g.gamma, f, pl, pr);
    else hllc_x_fp64(a, c, g.gamma, f, pl, pr);
    badL |= !(pos_finite(a[0]) && pos_finite(pl));
    badR |= !(pos_finite(c[0]) && pos_finite(pr));
  };
  // the Gauss points in mirror pairs (g, -g), each pair summed first: a
  // mirror image of the problem that reverses the points sums alike.  1D: one
  // point, twice half its flux.
#pragma unroll 1
  for (int kk = 0; kk < NS; ++kk) {
    double f1[4], f2[4];
    const int k2 = one ? kk : Q - 1 - kk;
    const double w = W.w[kk];
    if (k2 != kk) {
      point(kk, f1);
      point(k2, f2);
#pragma unroll
      for (int v = 0; v < 4; ++v) F[v] = fma(w, add_rn(f1[v], f2[v]), F[v]);
    } else {
      point(kk, f1);
#pragma unroll
      for (int v = 0; v < 4; ++v)
        F[v] = fma(w, one && R > 0 ? add_rn(f1[v], f1[v]) : f1[v], F[v]);
    }
    if (one) break;
  }
  const long long nf = d == 0 ? (long long)(g.nx + 1) * g.ny : (long long)g.nx * (g.ny + 1);
  const long long f = d == 0 ? (long long)j * (g.nx + 1) + i : (long long)j * g.nx + i;
  double* out = (d == 0 ? A.Fx : A.Fy) + f;
  out[0] = F[0];
  out[mn * nf] = F[1];
  out[mt * nf] = F[2];
  out[3 * nf] = F[3];
  (d == 0 ? A.fbx : A.fby)[f] = (uint8_t)((badL ? 1 : 0) | (badR ? 2 : 0));
  // a recorded step keeps the states for its adjoint
  if (double* tL = state_tape<double>(A, g, Q, d, 0)) {
    double* tR = state_tape<double>(A, g, Q, d, 1);
#pragma unroll 1
    for (int k = 0; k < 4 * Q; ++k) {
      const int v = k & 3, q = k >> 2;
      tL[((long long)v * Q + q) * nf + f] = L[(q * 4 + v) * lv];
      tR[((long long)v * Q + q) * nf + f] = M[(q * 4 + v) * kVar];
    }
  }
}

// the block's units blockIdx.x, + gridDim.x, ... of n.  unit(u, f): calls
// f(A, g, seg, r0, nb) for unit u, or not at all (nothing to do).  Both kinds
// of warps walk the same bands; band k of the walk uses buffer k % 2.
template <int R, class Unit>
__device__ __forceinline__ void faces_fx_block(const Unit& unit, const ParityW<double>& W, int n,
                                               int dirs, FxShared<R>& S) {
  const int warp = threadIdx.x >> 5;
  int k = 0;  // bands so far
  if (warp < 2 * kFxRows) {
    for (int u = blockIdx.x; u < n; u += gridDim.x)
      unit(u, [&](const StageArgs<double>& A, const Grid& g, int seg, int r0, int nb) {
        const int bands = unit_bands(g, r0, nb);
        for (int b = 0; b < bands; ++b, ++k) {
          if (k >= 2) bar_wait(3 + (k & 1));
          fx_produce<R>(A.X, g, W, seg, r0 - 1 + kFxRows * b, b == 0, dirs, S.band[k & 1],
                        S.top[k % 3]);
          bar_arrive(1 + (k & 1));
        }
      });
    // the arrivals on the empty barriers that no band waits for
    for (int m = k >= 2 ? k - 2 : 0; m < k; ++m) bar_wait(3 + (m & 1));
  } else {
    const int row = warp & 3, d = (warp >> 2) - 2;
    for (int u = blockIdx.x; u < n; u += gridDim.x)
      unit(u, [&](const StageArgs<double>& A, const Grid& g, int seg, int r0, int nb) {
        const int bands = unit_bands(g, r0, nb);
        for (int b = 0; b < bands; ++b, ++k) {
          bar_wait(1 + (k & 1));
          if ((dirs >> d) & 1) {
            const int j0 = r0 - 1 + kFxRows * b;
            if (g.riemann == 1)
              fx_solve<R, true>(A, g, W, seg, j0, b == 0, row, d, S.band[k & 1], S.top[(k + 2) % 3]);
            else
              fx_solve<R, false>(A, g, W, seg, j0, b == 0, row, d, S.band[k & 1], S.top[(k + 2) % 3]);
          }
          bar_arrive(3 + (k & 1));
        }
      });
  }
}

template <int R>
__global__ void __launch_bounds__(kFxThreads, 1) k_faces_fx(StageArgs<double> A, Grid g,
                                                           const __grid_constant__ ParityW<double> W,
                                                           int nseg, int nb, int units, int dirs) {
  pdl_wait();
  pdl_trigger();
  extern __shared__ __align__(16) unsigned char fx_smem[];
  faces_fx_block<R>(
      [&](int u, auto&& f) {
        const int chunk = u / nseg;
        f(A, g, u - chunk * nseg, chunk * (kFxRows * nb - 1), nb);
      },
      W, units, dirs, *reinterpret_cast<FxShared<R>*>(fx_smem));
}

// batches: a unit per item (problem, segment, first row, bands)
template <int R>
__global__ void __launch_bounds__(kFxThreads, 1) k_faces_fx_batch(
    StageArgs<double> B, const Prob* probs, const Scalars* psc, const Item* items, int nitems,
    const __grid_constant__ ParityW<double> W) {
  pdl_wait();
  pdl_trigger();
  extern __shared__ __align__(16) unsigned char fx_smem[];
  faces_fx_block<R>(
      [&](int u, auto&& f) {
        const Item w = items[u];
        if (psc[w.p].dt == 0.0) return;  // finished problem
        const Prob& P = probs[w.p];
        f(problem_args<double>(B, P, psc, w.p), P.g, w.a, w.b, w.pad);
      },
      W, nitems, 3, *reinterpret_cast<FxShared<R>*>(fx_smem));
}

}  // namespace gpm
