// weight_tables.h -- kernel weight tables from the binary128 solves: the
// full per-radius prediction vectors for the MOOD recompute and the parity
// coefficients of the top radius for the first pass.
#pragma once

#include <math.h>
#include <string.h>

#include "fixed_dot.h"
#include "gp_weights.h"
#include "gpmood_kernels.cuh"

namespace gpm {
namespace {

// index of offset (a,b) in the stencil order of gp_weights.c
int sidx(const gpw_radius& w, int a, int b) {
  for (int m = 0; m < w.n; ++m)
    if (w.da[m] == a && w.db[m] == b) return m;
  return -1;
}

// the prediction weight of stencil point (a, b) for face E, W, N, S and point
// k, from the east / north solves at g >= 0 by the mirrors: E at -g is E at
// g with b negated, W the x-mirror of E; N and S alike
double direct_weight(const gpw_radius& w, int face, int k, int a, int b) {
  const int kp = k < (w.q + 1) / 2 ? k : w.q - 1 - k;  // the +g point of the pair
  if (k != kp) (face < 2 ? b : a) *= -1;
  if (face == 1) a = -a;
  if (face == 3) b = -b;
  return w.z[face / 2][kp][sidx(w, a, b)];
}

// fixed-point bits T of a set of weights: the largest up to 60 that keeps
// every weight below one and every sum of |weight| below four
int weight_bits(double big, double l1) {
  int T = 60;
  while (T > 30 && (ldexp(big, T - 60) >= 1.0 - 0x1p-30 || ldexp(l1, T - 60) >= 3.9)) --T;
  return T;
}

// the parity coefficients cx, cy of the top radius, q points a face, in the
// form the face kernels read
void set_parity(const double (*cx)[kMaxN], const double (*cy)[kMaxN], const gpw_radius&,
                ParityW<float>& P) {
  for (int kk = 0; kk < 2; ++kk)
    for (int c = 0; c < kMaxN; ++c) {
      P.cx[kk][c] = (float)cx[kk][c];
      P.cy[kk][c] = (float)cy[kk][c];
    }
}
void set_parity(const double (*cx)[kMaxN], const double (*cy)[kMaxN], const gpw_radius& w,
                ParityW<double>& P) {
  double big = 0.0, l1 = 0.0;
  for (int kk = 0; kk < 2; ++kk)
    for (int c = 0; c < kMaxN; ++c)
      big = fmax(big, fmax(fabs(cx[kk][c]), fabs(cy[kk][c])));
  for (int face = 0; face < 2; ++face)
    for (int k = 0; k < w.q; ++k) {
      double s = 0.0;
      for (int m = 0; m < w.n; ++m) s += fabs(w.z[face][k][m]);
      l1 = fmax(l1, s);
    }
  const int R = w.q - 1;
  int T = weight_bits(big, l1) + 1;
  for (bool fits = false; !fits;) {
    --T;
    fits = true;
    for (int t = 0; t < 4; ++t) {
      const double* z = t < 2 ? cx[t] : cy[t - 2];
      int2* C = t < 2 ? P.cx[t] : P.cy[t - 2];
      fxd_load load[4] = {};  // of the sum of each parity
      for (int c = 0; c < kMaxN; ++c) {
        fxd_weight(z[c], T, &C[c].x, &C[c].y);
        if (c >= stencil_n(R)) continue;
        const Comp cm = comp_at(R, c);  // of 1, 2 or 4 cells
        fxd_count(&load[2 * cm.px + cm.py], C[c].x, C[c].y, (cm.a ? 2 : 1) * (cm.b ? 2 : 1));
      }
      for (int k = 0; k < 4; ++k) fits = fits && fxd_fits(&load[k]);
    }
  }
  P.off = 63 - T;
}

// the direct weights of every radius
template <class Real, class Table>
void plain_weights(const gpw_radius* wr, Table& D) {
  for (int R = 1; R <= 3; ++R)
    for (int face = 0; face < 4; ++face)
      for (int k = 0; k < wr[R].q && wr[R].n; ++k)
        for (int m = 0; m < wr[R].n; ++m)
          D.z[R][face][k][m] = (Real)direct_weight(wr[R], face, k, wr[R].da[m], wr[R].db[m]);
}
// the largest weight of any radius and the largest sum of |weight| of a point
void largest_weights(const gpw_radius* wr, double& big, double& l1) {
  for (int R = 1; R <= 3; ++R)
    for (int face = 0; face < 2; ++face)
      for (int k = 0; k < wr[R].q && wr[R].n; ++k) {
        double s = 0.0;
        for (int m = 0; m < wr[R].n; ++m) {
          s += fabs(wr[R].z[face][k][m]);
          big = fmax(big, fabs(wr[R].z[face][k][m]));
        }
        l1 = fmax(l1, s);
      }
}
void set_direct(const gpw_radius* wr, DirectW<float>& D) { plain_weights<float>(wr, D); }
void set_direct(const gpw_radius* wr, DirectW<double>& D) {
  double big = 0.0, l1 = 0.0;
  largest_weights(wr, big, l1);
  int T = weight_bits(big, l1) + 1;
  for (bool fits = false; !fits;) {
    --T;
    fits = true;
    for (int R = 1; R <= 3; ++R)
      for (int face = 0; face < 4; ++face)
        for (int k = 0; k < wr[R].q && wr[R].n; ++k) {
          fxd_load load = {0, 0, 0};
          for (int m = 0; m < wr[R].n; ++m) {
            const int a = wr[R].da[m], b = wr[R].db[m];
            int2& z = D.z[R][face][k][diamond3_slot(a, b)];
            fxd_weight(direct_weight(wr[R], face, k, a, b), T, &z.x, &z.y);
            fxd_count(&load, z.x, z.y, 1);
          }
          fits = fits && fxd_fits(&load);
        }
  }
  D.off = 63 - T;
}

void fill_gather(const gpw_radius* wr, int top, GatherW<float>& G) {
  memset(&G, 0, sizeof(G));
  G.top = top;
  plain_weights<float>(wr, G);
}
void fill_gather(const gpw_radius* wr, int top, GatherW<double>& G) {
  memset(&G, 0, sizeof(G));
  G.top = top;
  double big = 0.0, l1 = 1.0;
  largest_weights(wr, big, l1);
  // a cell's sum over its neighbours' faces (4 q values each, every face at a
  // radius of its own) stays below 2^63 of the products' high limbs
  int T = 58;
  while (T > 30 && (ldexp(big, T - 58) > 1.0 || ldexp(l1, T - 58) >= 3.9)) --T;
  ++T;
  for (bool fits = false; !fits;) {
    --T;
    fits = true;
    for (int face = 0; face < 4; ++face) {
      int2& c = G.z[0][face][0][diamond3_slot(0, 0)];
      fxd_weight(1.0, T, &c.x, &c.y);
    }
    for (int R = 1; R <= 3; ++R)
      for (int face = 0; face < 4; ++face)
        for (int k = 0; k < wr[R].q && wr[R].n; ++k)
          for (int m = 0; m < wr[R].n; ++m) {
            const int a = wr[R].da[m], b = wr[R].db[m];
            int2& z = G.z[R][face][k][diamond3_slot(a, b)];
            fxd_weight(direct_weight(wr[R], face, k, a, b), T, &z.x, &z.y);
          }
    // the limbs of one neighbour's sum: of each face the radius with the most
    for (int slot = 0; slot < kMaxN; ++slot) {
      fxd_load load = {0, 0, 0};
      for (int face = 0; face < 4; ++face) {
        fxd_load most = {0, 0, 0};
        for (int R = 0; R <= 3; ++R) {
          fxd_load one = {0, 0, 0};
          for (int k = 0; k < kMaxQ; ++k)
            fxd_count(&one, G.z[R][face][k][slot].x, G.z[R][face][k][slot].y, 1);
          most = {fmax(most.mid, one.mid), fmax(most.up, one.up), fmax(most.down, one.down)};
        }
        load = {load.mid + most.mid, load.up + most.up, load.down + most.down};
      }
      fits = fits && fxd_fits(&load);
    }
  }
  G.off = 65 - T;
}

template <class Real>
void fill_weights(const gpw_radius* wr, int top, const double* d2x, const double* d2y,
                  ParityW<Real>& P, DirectW<Real>& D) {
  memset(&P, 0, sizeof(P));
  memset(&D, 0, sizeof(D));
  D.top = top;
  D.w[0][0] = Real(1);
  for (int m = 0; m < 5; ++m) {
    D.d2x[m] = (Real)d2x[m];
    D.d2y[m] = (Real)d2y[m];
  }
  for (int R = 1; R <= 3; ++R)
    for (int k = 0; k < wr[R].q && wr[R].n; ++k) D.w[R][k] = (Real)wr[R].w[k];
  set_direct(wr, D);
  // parity coefficients of the top radius
  const int R = top;
  if (R == 0) {  // the face states are the cell averages
    P.w[0] = Real(1);
    return;
  }
  double cx[2][kMaxN], cy[2][kMaxN];
  memset(cx, 0, sizeof(cx));
  memset(cy, 0, sizeof(cy));
  const gpw_radius& w = wr[R];
  const int q = w.q, ns = (q + 1) / 2;
  for (int k = 0; k < q; ++k) P.w[k] = (Real)w.w[k];
  for (int kk = 0; kk < ns; ++kk) {
    const bool middle = (q & 1) && kk == q / 2;
    for (int c = 0; c < stencil_n(R); ++c) {
      Comp cm = comp_at(R, c);
      double ex = 0.0, ny = 0.0;
      int cnt = 0;
      for (int sa = 1; sa >= -1; sa -= 2) {
        if (cm.a == 0 && sa < 0) continue;
        for (int sb = 1; sb >= -1; sb -= 2) {
          if (cm.b == 0 && sb < 0) continue;
          double chi = (cm.px && sa < 0 ? -1.0 : 1.0) * (cm.py && sb < 0 ? -1.0 : 1.0);
          ex += chi * w.z[0][kk][sidx(w, sa * cm.a, sb * cm.b)];
          ny += chi * w.z[1][kk][sidx(w, sa * cm.a, sb * cm.b)];
          ++cnt;
        }
      }
      ex /= cnt;
      ny /= cnt;
      // at g = 0 the odd components across the face vanish exactly
      if (middle && cm.py) ex = 0.0;
      if (middle && cm.px) ny = 0.0;
      cx[kk][c] = ex;
      cy[kk][c] = ny;
    }
  }
  set_parity(cx, cy, w, P);
}

}  // namespace
}  // namespace gpm
