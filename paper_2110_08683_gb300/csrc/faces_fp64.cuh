// faces_fp64.cuh -- first-pass faces at the top radius, FP64.
//
// What bounds it: the FP64 pipe (64 cycles a warp instruction a
// sub-partition) in the Riemann solver, the integer pipes in the
// reconstruction (fixed_dot.h).  Three blocks an SM keep both busy: while
// one block solves, another reconstructs.  4096 x 1024 double Mach
// reflection, R = 3: 4.6 ms a launch.  It was 11.1 ms with everything on the
// FP64 pipe (716 FP64 instructions a face) and 6.0 ms with the
// reconstruction's 396 taken off it; the solver now takes 180 for 320.
#pragma once

#include "gpmood_kernels.cuh"

namespace gpm {

// A block of 4 warps walks up a segment of 32 cell columns in bands of 4
// rows.  Per band, lane l and warp w hold cell (i0 + l, j + w),
// i0 = 31 seg - 1: the cell's parity sums give its states on all four faces
// (shared memory), then the thread solves the x face to its left and the y
// face below it.  The upper states of a band's last row stay for the next
// band, so that every warp has faces to solve in every band but the first,
// whose row 0 only supplies states: FP64 work is spread evenly over the four
// sub-partitions (a block of 8 rows that owns 7 leaves one of them half
// idle).
constexpr int kFxRows = 4;

template <int R>
struct FxShared {
  static constexpr int Q = rule_q(R);
  double x[2][Q][4][kFxRows][32];   // [east, west][point][variable][row][lane]
  double n[Q][4][kFxRows + 1][32];  // north; row 0: the last row of the band before
  double s[Q][4][kFxRows][32];      // south
};

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

// faces of segment seg, rows r0 .. r0 + 4 nb - 2 (x faces of rows below ny, y
// faces up to ny); dirs: 1 x faces, 2 y faces, 3 both
template <int R>
__device__ __forceinline__ void faces_fx_block(const StageArgs<double>& A, const Grid& g,
                                               const ParityW<double>& W, int seg, int r0, int nb,
                                               int dirs, FxShared<R>& S) {
  constexpr int Q = rule_q(R);
  constexpr int NS = (Q + 1) / 2;
  constexpr int kVar = kFxRows * 32, kVarN = (kFxRows + 1) * 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int i = seg * kSegFaces - 1 + lane, ic = i < g.nx ? i : g.nx;
  // the 1D method's points all carry the same state: one pair is formed, one
  // point solved
  const bool one = g.dim == 1;
  const int npair = one ? 1 : NS;
#pragma unroll 1
  for (int b = 0; b < nb; ++b) {
    const int j0 = r0 - 1 + kFxRows * b, j = j0 + warp;
    if (j0 > g.ny) break;                  // whole block
    const bool owned = b > 0 || warp > 0;  // this row's faces are the block's
    const bool xrow = (dirs & 1) && owned && j < g.ny;
    const bool ystate = (dirs & 2) && j <= g.ny;
    if (b > 0 && warp == kFxRows - 1) {
#pragma unroll
      for (int k = 0; k < 4 * Q; ++k) S.n[k >> 2][k & 3][0][lane] = S.n[k >> 2][k & 3][kFxRows][lane];
    }
    if (xrow || ystate) {
      const double* X = A.X + (long long)(j + g.H) * g.pitch + (ic + g.H);
      const int pitch = g.pitch;
#pragma unroll 1
      for (int v = 0; v < 4; ++v, X += g.vstride) {
        double* xe = &S.x[0][0][v][warp][lane];
        double* xw = &S.x[1][0][v][warp][lane];
        double* yn = &S.n[0][v][warp + 1][lane];
        double* ys = &S.s[0][v][warp][lane];
        if constexpr (R == 0) {
          const double u = __ldg(X);
          *xe = *xw = u;
          *yn = *ys = u;
        } else {
          ReconFixed<R> rc;
          rc.sums([&](int a, int c) -> double { return __ldg(X + (long long)c * pitch + a); },
                  true);
          if (xrow) fx_states<R, 0>(rc, W, npair, xe, 4 * kVar, xw, 4 * kVar);
          if (ystate) fx_states<R, 1>(rc, W, npair, yn, 4 * kVarN, ys, 4 * kVar);
        }
      }
    }
    __syncthreads();
    if (owned && lane >= 1) {
#pragma unroll 1
      for (int d = 0; d < 2; ++d) {
        // x face between (i-1, j) and (i, j); y face between (i, j-1) and (i, j)
        if (!((dirs >> d) & 1) || (d == 0 ? (j >= g.ny || i > g.nx) : (j > g.ny || i >= g.nx)))
          continue;
        const double* L = d == 0 ? &S.x[0][0][0][warp][lane - 1] : &S.n[0][0][warp][lane];
        const double* M = d == 0 ? &S.x[1][0][0][warp][lane] : &S.s[0][0][warp][lane];
        const int lv = d == 0 ? kVar : kVarN;  // variable strides; points four apart
        const int mn = 1 + d, mt = 2 - d;      // normal and tangential momentum
        double F[4] = {0, 0, 0, 0};            // mass, normal, tangential, energy
        bool badL = false, badR = false;
        auto point = [&](int q, double* f) {
          const double* l = L + q * 4 * lv;
          const double* m = M + q * 4 * kVar;
          const double a[4] = {l[0], l[mn * lv], l[mt * lv], l[3 * lv]};
          const double c[4] = {m[0], m[mn * kVar], m[mt * kVar], m[3 * kVar]};
          double pl, pr;
          riemann_x<double>(g.riemann, a, c, g.gamma, f, pl, pr);
          badL |= !(pos_finite(a[0]) && pos_finite(pl));
          badR |= !(pos_finite(c[0]) && pos_finite(pr));
        };
        // the Gauss points in mirror pairs (g, -g), each pair summed first: a
        // mirror image of the problem that reverses the points sums alike
#pragma unroll 1
        for (int kk = 0; kk < npair; ++kk) {
          const double w = W.w[kk];
          double f1[4], f2[4] = {0, 0, 0, 0};
          point(kk, f1);
          const int k2 = Q - 1 - kk;
          if (one) {
#pragma unroll
            for (int v = 0; v < 4; ++v) f2[v] = f1[v];
          } else if (k2 != kk) {
            point(k2, f2);
          }
#pragma unroll
          for (int v = 0; v < 4; ++v)
            F[v] = fma(w, (one || k2 != kk) ? add_rn(f1[v], f2[v]) : f1[v], F[v]);
        }
        const uint8_t bits = (uint8_t)((badL ? 1 : 0) | (badR ? 2 : 0));
        const long long nf = d == 0 ? (long long)(g.nx + 1) * g.ny : (long long)g.nx * (g.ny + 1);
        const long long f = d == 0 ? (long long)j * (g.nx + 1) + i : (long long)j * g.nx + i;
        double* out = (d == 0 ? A.Fx : A.Fy) + f;
        out[0] = F[0];
        out[mn * nf] = F[1];
        out[mt * nf] = F[2];
        out[3 * nf] = F[3];
        (d == 0 ? A.fbx : A.fby)[f] = bits;
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
    }
    __syncthreads();
  }
}

template <int R>
__global__ void __launch_bounds__(32 * kFxRows, 3) k_faces_fx(StageArgs<double> A, Grid g,
                                                             const __grid_constant__ ParityW<double> W,
                                                             int nseg, int nb, int dirs) {
  pdl_wait();
  pdl_trigger();
  extern __shared__ __align__(16) unsigned char fx_smem[];
  const int chunk = blockIdx.x / nseg;
  faces_fx_block<R>(A, g, W, blockIdx.x - chunk * nseg, chunk * (kFxRows * nb - 1), nb, dirs,
                    *reinterpret_cast<FxShared<R>*>(fx_smem));
}

// batches: one block per item (problem, segment, first row, bands)
template <int R>
__global__ void __launch_bounds__(32 * kFxRows, 3) k_faces_fx_batch(
    StageArgs<double> B, const Prob* probs, const Scalars* psc, const Item* items,
    const __grid_constant__ ParityW<double> W) {
  pdl_wait();
  pdl_trigger();
  extern __shared__ __align__(16) unsigned char fx_smem[];
  // the item's problem, read from shared memory on demand like kernel
  // parameters
  __shared__ Prob sp;
  __shared__ StageArgs<double> sa;
  __shared__ Item sw;
  __shared__ int done;
  if (threadIdx.x == 0) {
    sw = items[blockIdx.x];
    sp = probs[sw.p];
    sa = problem_args<double>(B, sp, psc, sw.p);
    done = psc[sw.p].dt == 0.0;  // finished problem
  }
  __syncthreads();
  if (done) return;  // uniform over the block
  faces_fx_block<R>(sa, sp.g, W, sw.a, sw.b, sw.pad, 3,
                    *reinterpret_cast<FxShared<R>*>(fx_smem));
}

}  // namespace gpm
