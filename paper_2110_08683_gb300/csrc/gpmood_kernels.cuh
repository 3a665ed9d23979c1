// gpmood_kernels.cuh -- CUDA kernels of the GP-MOOD stage (sm_103a).
//
// One RK stage (Sec. 4, Steps 3-10) of a single problem runs as
//   fill_ghosts -> faces -> update_first                  (first pass, all cells)
//   mood_loop                                             (troubled cells only)
// faces (FP64: faces_fp64.cuh; FP32: k_faces_xy, or k_faces a direction)
// reconstruct the pointwise Riemann states of eq. gp_reconstructor at the Gauss
// points of Table QR, apply face-state CAD (Sec. 3.3.1), solve HLLC and store
// the face-averaged flux of eq. fvm_F.
// update_first forms the candidate of eq. fvm_discrete, runs Steps 4-9,
// writes the SSP-RK3 combination (eq. rk3) and appends troubled cells to a
// queue with one atomic per warp.  mood_loop iterates on the device, with
// barriers between its phases among as many blocks as the queue is worth: it
// lowers the order of queued cells
// by one cascade level, recomputes the faces whose EDP1 order changed (Sec.
// 3.6) and re-updates + re-detects the queued cells and their face
// neighbours, until no cell is troubled.  Batches run the same kernels over the
// work items and the pooled queue of many problems.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "gpmood_internal.h"
#include "fixed_dot.h"
#include "fp_bits.h"
#include "fp_newton.h"
#include "spin_limit.h"

namespace gpm {

// ---------------------------------------------------------------------------
// indexing
// ---------------------------------------------------------------------------
__device__ __forceinline__ long long gidx(const Grid& g, int v, int i, int j) {
  return (long long)v * g.vstride + (long long)(j + g.H) * g.pitch + (i + g.H);
}
// x-face i (0..nx) of row j: between cells i-1 and i
__device__ __forceinline__ long long fxidx(const Grid& g, int v, int i, int j) {
  return ((long long)v * g.ny + j) * (g.nx + 1) + i;
}
// y-face j (0..ny) of column i: between cells j-1 and j
__device__ __forceinline__ long long fyidx(const Grid& g, int v, int i, int j) {
  return ((long long)v * (g.ny + 1) + j) * g.nx + i;
}
__device__ __forceinline__ int cidx(const Grid& g, int i, int j) { return j * g.nx + i; }

__device__ __forceinline__ int wrapi(int i, int n) {
  int r = i % n;
  return r < 0 ? r + n : r;
}

// ---------------------------------------------------------------------------
// stencil algebra at compile time.
// The blocky diamond |a|+|b| <= R is invariant under x -> -x and y -> -y, and
// so is the SE kernel; hence the west-face weights are the x-mirror of the
// east-face ones, the point -g the mirror of +g, and the same for north /
// south.  Grouping the stencil into mirror orbits {(+-a, +-b)} and using the
// even/odd combinations of each orbit ("parity sums") turns the 2q face
// states of one axis into q dot products of length N plus butterflies,
// instead of 2q dot products.  The parity sums of one cell are shared by all
// four faces.
// ---------------------------------------------------------------------------
__host__ __device__ constexpr int stencil_n(int R) { return 2 * R * R + 2 * R + 1; }
__host__ __device__ constexpr int rule_q(int R) { return R == 0 ? 1 : R + 1; }

struct Comp {
  int a, b, px, py;
};

// k-th parity component: reps (a,b) with a,b >= 0, a+b <= R in order b-major,
// and for each rep the types ee, oe (a>0), eo (b>0), oo (a,b>0)
__host__ __device__ constexpr Comp comp_at(int R, int k) {
  int n = 0;
  for (int b = 0; b <= R; ++b)
    for (int a = 0; a + b <= R; ++a) {
      if (n == k) return Comp{a, b, 0, 0};
      ++n;
      if (a > 0) {
        if (n == k) return Comp{a, b, 1, 0};
        ++n;
      }
      if (b > 0) {
        if (n == k) return Comp{a, b, 0, 1};
        ++n;
      }
      if (a > 0 && b > 0) {
        if (n == k) return Comp{a, b, 1, 1};
        ++n;
      }
    }
  return Comp{0, 0, 0, 0};
}

// parity sums of one variable around a cell; ld(a, b) loads the cell (i+a, j+b)
template <int R, class Real, class Load>
__device__ __forceinline__ void parity_sums(const Load& ld, Real* s) {
  int k = 0;
#pragma unroll
  for (int b = 0; b <= R; ++b) {
#pragma unroll
    for (int a = 0; a + b <= R; ++a) {
      if (a == 0 && b == 0) {
        s[k++] = ld(0, 0);
      } else if (b == 0) {
        Real p = ld(a, 0), m = ld(-a, 0);
        s[k++] = p + m;
        s[k++] = p - m;
      } else if (a == 0) {
        Real p = ld(0, b), m = ld(0, -b);
        s[k++] = p + m;
        s[k++] = p - m;
      } else {
        Real q1 = ld(a, b), q2 = ld(-a, b), q3 = ld(a, -b), q4 = ld(-a, -b);
        Real p1 = q1 + q2, m1 = q1 - q2, p2 = q3 + q4, m2 = q3 - q4;
        s[k++] = p1 + p2;  // ee
        s[k++] = m1 + m2;  // oe
        s[k++] = p1 - p2;  // eo
        s[k++] = m1 - m2;  // oo
      }
    }
  }
}

// the face states of one variable of one cell from its parity sums: sums()
// takes the stencil in, dot() forms the sums T[px][py] over the components
// of each parity, whose sums and differences (the butterflies) are the face
// states, and out() turns one into a Real.  dead: no cell here, all sums zero.
template <int R, class Real>
struct Recon {
  using T = Real;
  Real s[stencil_n(R)];
  template <class Load>
  __device__ __forceinline__ void sums(const Load& ld, bool live) {
    if (live) {
      parity_sums<R, Real>(ld, s);
    } else {
#pragma unroll
      for (int k = 0; k < stencil_n(R); ++k) s[k] = Real(0);
    }
  }
  // R = 0: the face states are the cell average itself
  template <class Coef>
  __device__ __forceinline__ void dot(const Coef* c, Real t[2][2]) const {
    t[0][0] = t[0][1] = t[1][0] = t[1][1] = Real(0);
    if (R == 0) {
      t[0][0] = s[0];
      return;
    }
    if constexpr (R > 0) {
#pragma unroll
      for (int k = 0; k < stencil_n(R); ++k) {
        const Comp cm = comp_at(R, k);
        t[cm.px][cm.py] = fma(c[k], s[k], t[cm.px][cm.py]);
      }
    }
  }
  __device__ __forceinline__ Real out(Real t, const ParityW<Real>&) const { return t; }
};

// FP64, R > 0: in fixed point on the integer pipes (fixed_dot.h), scaled by
// the largest exponent of the cell's own stencil, so that a face state
// depends on its stencil alone and not on the tile it was computed in.
template <int R>
struct ReconFixed {
  using T = long long;
  int2 s[stencil_n(R)];  // limbs of the parity sums (x high, y low)
  int E;                 // reference exponent
  uint32_t special;      // NaN bits: the stencil holds a NaN or an infinity
  template <class Load>
  __device__ __forceinline__ void sums(const Load& ld, bool live) {
    double x[stencil_n(R)];
    int k = 0;
#pragma unroll
    for (int b = -R; b <= R; ++b)
#pragma unroll
      for (int a = -R; a <= R; ++a)
        if ((a < 0 ? -a : a) + (b < 0 ? -b : b) <= R) x[k++] = live ? ld(a, b) : 0.0;
    uint32_t top = (uint32_t)FXD_EMIN << 20;
#pragma unroll
    for (int m = 0; m < stencil_n(R); ++m) top = max(top, fxd_hi(x[m]) & 0x7fffffffu);
    E = (int)(top >> 20);
    special = E == 0x7ff ? 0x7ff80000u : 0u;
    long long X[stencil_n(R)], p[stencil_n(R)];
#pragma unroll
    for (int m = 0; m < stencil_n(R); ++m) X[m] = fxd_from_double(x[m], E);
    auto at = [&](int a, int b) -> long long {
      int m = 0;
      for (int bb = -R; bb < b; ++bb) m += 2 * (R - (bb < 0 ? -bb : bb)) + 1;
      return X[m + a + R - (b < 0 ? -b : b)];
    };
    parity_sums<R, long long>(at, p);
#pragma unroll
    for (int m = 0; m < stencil_n(R); ++m) s[m] = make_int2(fxd_limb_hi(p[m]), fxd_limb_lo(p[m]));
  }
  __device__ __forceinline__ void dot(const int2* c, long long t[2][2]) const {
    fxd_acc acc[2][2] = {};
#pragma unroll
    for (int k = 0; k < stencil_n(R); ++k) {
      const Comp cm = comp_at(R, k);
      fxd_mac(&acc[cm.px][cm.py], c[k].x, c[k].y, s[k].x, s[k].y);
    }
#pragma unroll
    for (int px = 0; px < 2; ++px)
#pragma unroll
      for (int py = 0; py < 2; ++py) t[px][py] = fxd_round(acc[px][py]);
  }
  __device__ __forceinline__ double out(long long t, const ParityW<double>& W) const {
    return fxd_to_double(t, E, W.off, special);
  }
};
template <>
struct Recon<1, double> : ReconFixed<1> {};
template <>
struct Recon<2, double> : ReconFixed<2> {};
template <>
struct Recon<3, double> : ReconFixed<3> {};

// ---------------------------------------------------------------------------
// Euler equations (eq. euler_eqn) and HLLC (Toro et al. 1994) in Real
// ---------------------------------------------------------------------------
template <class Real>
__device__ __forceinline__ Real pressure_of(const Real* U, Real gm1) {
  Real ir = Real(1) / U[0];
  return gm1 * (U[3] - Real(0.5) * (U[1] * U[1] + U[2] * U[2]) * ir);
}

// finite (neither infinite nor NaN), decided on the bit pattern
__device__ __forceinline__ bool finite_r(double x) {
  return (__double_as_longlong(x) & 0x7fffffffffffffffll) < 0x7ff0000000000000ll;
}
__device__ __forceinline__ bool finite_r(float x) { return isfinite(x); }

// reciprocal from the hardware approximation r (rcp.approx.ftz.f64, whose
// relative error stays below 2^-20 on this GPU): with e = 1 - x r,
// 1/x = r / (1 - e) = r (1 + e + e^2 + ...), and the series cut after e^2
// leaves a relative error below 2^-60 before the final rounding (one FMA
// fewer than two Newton-Raphson steps).  FP32: rcp.approx.ftz.f32 (within 1
// ulp) and one Newton-Raphson step r + r (1 - x r).  Zero or non-finite x
// give a non-finite result.
__device__ __forceinline__ double recip(double x) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  const double e = fma(-x, r, 1.0);
  return fma(r, fma(e, e, e), r);
}
__device__ __forceinline__ float recip(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return fmaf(r, fmaf(-x, r, 1.0f), r);
}

// square root of a sound-speed argument z > 0, FP32: the hardware
// approximation sqrt.approx.ftz.f32 (the FP32 path's reconstruction and
// Riemann solver are FP32 arithmetic throughout)
__device__ __forceinline__ float sqrt_r(float x) {
  float r;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// products and sums rounded one by one (no contraction into an FMA): where
// an expression's mirror image swaps its terms, both then round alike, so a
// mirror-symmetric problem stays symmetric bit for bit
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }

// pressure of a conservative state with 1/rho given, the velocities out: one
// fixed sequence of rounded operations, so two states that are mirror images
// (a momentum component negated) give the same pressure bit for bit, whichever
// side of a face or of a cell each sits on
template <class Real>
__device__ __forceinline__ Real pressure_ir(const Real* U, Real ir, Real gm1, Real& u, Real& v) {
  u = mul_rn(U[1], ir);
  v = mul_rn(U[2], ir);
  const Real k = fma(U[1], u, mul_rn(U[2], v));  // m_x u + m_y v
  return mul_rn(gm1, fma(Real(-0.5), k, U[3]));
}

// quiet NaN: the flux of a face whose state lies outside the Riemann solver's
// domain (non-positive or non-finite density or pressure) is undefined
__device__ __forceinline__ void qnan(double& x) { x = __longlong_as_double(0x7ff8000000000000ll); }
__device__ __forceinline__ void qnan(float& x) { x = __int_as_float(0x7fc00000); }
// x > 0 and finite, decided on the integer bits (positive finite values are
// the bit patterns strictly between +0 and +inf; NaN and negatives fall
// outside): the same answer as the two comparisons without denormal
// flushing, taken off the floating-point pipes
__device__ __forceinline__ bool pos_finite(double x) {
  const long long b = __double_as_longlong(x);
  return b > 0 && b < 0x7ff0000000000000ll;
}
__device__ __forceinline__ bool pos_finite(float x) {
  const int b = __float_as_int(x);
  return b > 0 && b < 0x7f800000;
}
// comparisons of doubles on the integer pipes (fp_bits.h: the IEEE answer
// exactly, for the inputs each name allows).  An FP64 compare, min or max
// occupies the FP64 pipe like an FMA does (on this GPU about 64 cycles per
// warp instruction per sub-partition), a 64-bit integer compare a few
// cycles.  FP32 keeps the hardware compare, which is cheap.
__device__ __forceinline__ bool is_nan(double x) { return fpb_is_nan(x); }
// a < b, a and b not NaN
__device__ __forceinline__ bool lt_num(double a, double b) { return fpb_lt_num(a, b); }
__device__ __forceinline__ bool lt_num(float a, float b) { return a < b; }
// a < b with NaN (false when either is NaN)
__device__ __forceinline__ bool lt_ieee(double a, double b) { return fpb_lt_ieee(a, b); }
__device__ __forceinline__ bool lt_ieee(float a, float b) { return a < b; }
// a <= b with NaN (false when either is NaN)
__device__ __forceinline__ bool le_ieee(double a, double b) { return fpb_le_ieee(a, b); }
__device__ __forceinline__ bool le_ieee(float a, float b) { return a <= b; }
// x >= 0 and x > 0, x not NaN
__device__ __forceinline__ bool ge0_num(double x) { return fpb_ge0_num(x); }
__device__ __forceinline__ bool ge0_num(float x) { return x >= 0.0f; }
__device__ __forceinline__ bool gt0_num(double x) { return fpb_gt0_num(x); }
__device__ __forceinline__ bool gt0_num(float x) { return x > 0.0f; }
// a < b ? a : b and a > b ? a : b, a and b not NaN
template <class Real>
__device__ __forceinline__ Real min_num(Real a, Real b) { return lt_num(a, b) ? a : b; }
template <class Real>
__device__ __forceinline__ Real max_num(Real a, Real b) { return lt_num(b, a) ? a : b; }

template <class Real>
__device__ __forceinline__ bool solver_domain(Real rL, Real rR, Real pL, Real pR) {
  // rho > 0 and p > 0 (non-finite inputs give a NaN flux anyway)
  return pos_finite(rL) && pos_finite(rR) && pos_finite(pL) && pos_finite(pR);
}

// x-direction HLLC flux; pL/pR return the pressures of the two states so the
// caller can run face-state CAD without another EoS evaluation.
// wave speeds S_L = min(uL-cL, uR-cR), S_R = max(uL+cL, uR+cR); the star
// state is taken on the side of the contact speed S*.  Every product is an
// explicit fma or a product rounded on its own, so the compiler cannot fuse
// operations differently in different kernels: every kernel that solves a
// face gets the same flux bit for bit.  Inside the solver's domain every
// value is finite, so the comparisons run on the integer pipes (outside it
// the flux is NaN whatever they decide).
template <class Real>
__device__ __forceinline__ void hllc_x(const Real* UL, const Real* UR, Real gam, Real* F,
                                       Real& pL, Real& pR) {
  const Real gm1 = gam - Real(1);
  Real rL = UL[0], rR = UR[0];
  Real irL = recip(rL), irR = recip(rR);
  Real uL, vL, uR, vR;
  pL = pressure_ir(UL, irL, gm1, uL, vL);
  pR = pressure_ir(UR, irR, gm1, uR, vR);
  Real cL = sqrt_r(mul_rn(mul_rn(gam, pL), irL)), cR = sqrt_r(mul_rn(mul_rn(gam, pR), irR));
  const Real SL = min_num(uL - cL, uR - cR);
  const Real SR = max_num(uL + cL, uR + cR);
  Real dL = SL - uL, dR = SR - uR;
  const Real mL = mul_rn(rL, uL), mR = mul_rn(rR, uR);
  Real num = fma(-mR, dR, fma(mL, dL, pR - pL));
  Real den = fma(-rR, dR, mul_rn(rL, dL));
  Real Ss = mul_rn(num, recip(den));
  const bool left = ge0_num(Ss);
  const bool useL = ge0_num(SL);
  const bool useS = left || gt0_num(SR);
  // star state on side K of the contact: with m = rho_K (S_K - u_K) and
  // D = 1 / (S_K - S*), rho* = m D and
  //   (rho E)* = rho* (E_K/rho_K + (S* - u_K)(S* + p_K / m))
  //            = D ((S_K - u_K) E_K + (S* - u_K)(m S* + p_K)),
  // the second form needing no reciprocal of rho_K (S_K - u_K)
  Real rK = left ? rL : rR, uK = left ? uL : uR, vK = left ? vL : vR;
  Real EK = left ? UL[3] : UR[3], pK = left ? pL : pR, SK = left ? SL : SR;
  Real dK = left ? dL : dR;
  const Real m = mul_rn(rK, dK), iD = recip(SK - Ss);
  Real fK = mul_rn(m, iD);
  Real UKs[4] = {fK, mul_rn(fK, Ss), mul_rn(fK, vK),
                 mul_rn(iD, fma(dK, EK, mul_rn(Ss - uK, fma(m, Ss, pK))))};
  // one physical flux is ever used: F_L when S_L >= 0, F_R when S_R <= 0,
  // else the star flux F_K + S_K (U*_K - U_K) on side K
  const bool sideL = useL || (useS && left);
  const Real uX = sideL ? uL : uR, vX = sideL ? vL : vR, pX = sideL ? pL : pR;
  const Real mX = sideL ? mL : mR, EX = sideL ? UL[3] : UR[3];
  const Real FX[4] = {mX, fma(mX, uX, pX), mul_rn(mX, vX), mul_rn(uX, EX + pX)};
  const bool star = !useL && useS;
  const bool dom = solver_domain(rL, rR, pL, pR);
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    const Real UK = left ? UL[v] : UR[v];
    F[v] = star ? fma(SK, UKs[v] - UK, FX[v]) : FX[v];
    if (!dom) qnan(F[v]);
  }
}

// x-direction HLL flux (Harten, Lax and van Leer 1983): the single
// intermediate state between the wave speeds of hllc_x; pL/pR as there
template <class Real>
__device__ __forceinline__ void hll_x(const Real* UL, const Real* UR, Real gam, Real* F,
                                      Real& pL, Real& pR) {
  const Real gm1 = gam - Real(1);
  Real rL = UL[0], rR = UR[0];
  Real irL = recip(rL), irR = recip(rR);
  Real uL, vL, uR, vR;
  pL = pressure_ir(UL, irL, gm1, uL, vL);
  pR = pressure_ir(UR, irR, gm1, uR, vR);
  Real cL = sqrt_r(mul_rn(mul_rn(gam, pL), irL)), cR = sqrt_r(mul_rn(mul_rn(gam, pR), irR));
  const Real SL = min_num(uL - cL, uR - cR);
  const Real SR = max_num(uL + cL, uR + cR);
  // physical fluxes by the same rounded sequence on both sides
  const Real mL = mul_rn(rL, uL), mR = mul_rn(rR, uR);
  Real FL[4] = {mL, fma(mL, uL, pL), mul_rn(mL, vL), mul_rn(uL, UL[3] + pL)};
  Real FR[4] = {mR, fma(mR, uR, pR), mul_rn(mR, vR), mul_rn(uR, UR[3] + pR)};
  const Real iw = recip(SR - SL);
  const bool useL = ge0_num(SL), useR = !gt0_num(SR);
  const bool dom = solver_domain(rL, rR, pL, pR);
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    // x-mirror: (L, R, S_L, S_R) -> (R', L', -S_R, -S_L) swaps the two
    // products; each is rounded on its own so the mirror face negates exactly
    const Real a = mul_rn(SR, FL[v]), b = mul_rn(SL, FR[v]);
    const Real c = mul_rn(mul_rn(SL, SR), UR[v] - UL[v]);
    Real Fm = add_rn(a - b, c) * iw;
    F[v] = useL ? FL[v] : (useR ? FR[v] : Fm);
    if (!dom) qnan(F[v]);
  }
}

// ---------------------------------------------------------------------------
// the same two solvers in FP64.  Every FP64 instruction of a warp costs a
// sub-partition 64 cycles, so they are written for few of them: 41 an HLLC
// point (76 as hllc_x above, whose reciprocals and roots took 24):
//  - reciprocals and square roots on the integer pipes (fp_newton.h);
//  - products rho u are the momenta themselves;
//  - one flux formula f = (f0, f0 u + p, f0 v, u H) for the star region, whose
//    velocity is the contact's, u = S*, and for the physical flux of a side,
//    which is what u = u_K makes of it: with d_K = S_K - u_K, q_K = rho_K d_K
//    (Rankine-Hugoniot across S_K)
//      p = p_K + q_K (u - u_K), f0 = q_K / (S_K - u) u (or the momentum itself),
//      H = E + p = (d_K E_K + p S_K - p_K u_K) / (S_K - u).
// All products and sums are rounded one by one or explicit FMAs, so every
// kernel gets the same flux bit for bit.
// ---------------------------------------------------------------------------
__device__ __forceinline__ double recip_int(double x) {
  float s;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(s) : "f"(fpn_recip_arg(x)));
  return fpn_recip_seeded(x, s);
}
__device__ __forceinline__ double sqrt_int(double z) {
  float s;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(s) : "f"(fpn_sqrt_arg(z)));
  return fpn_sqrt_seeded(z, s);
}
// x / 2 for |x| >= 2^-1021 (its exponent reduced)
__device__ __forceinline__ double half_of(double x) {
  return __longlong_as_double(__double_as_longlong(x) - (1ll << 52));
}
// positive, finite and normal: the arguments recip_int and sqrt_int take
__device__ __forceinline__ bool pos_normal(double x) {
  const long long b = __double_as_longlong(x);
  return b >= 0x0010000000000000ll && b < 0x7ff0000000000000ll;
}

// one side of a face: velocities, twice the kinetic energy, pressure, sound
// speed and 1/rho
struct Side {
  double u, v, k, p, c, ir;
  bool ok;  // inside the solver's domain
};
__device__ __forceinline__ Side side_of(const double* U, double gam, double gm1) {
  Side s;
  s.ir = recip_int(U[0]);
  s.u = __dmul_rn(U[1], s.ir);
  // by the velocities, although (m_x^2 + m_y^2) / rho is a product less where v
  // has no other use: squares of momenta leave the range of doubles long before
  // the state does (below 1e-154 and above 1e154)
  s.v = __dmul_rn(U[2], s.ir);
  s.k = fma(U[1], s.u, __dmul_rn(U[2], s.v));
  s.p = __dmul_rn(gm1, fma(-0.5, s.k, U[3]));
  s.ok = pos_normal(U[0]) && pos_normal(s.p);
  s.c = sqrt_int(__dmul_rn(__dmul_rn(gam, s.p), s.ir));
  // what the caller checks: outside the domain the pressure is not a number
  if (!pos_normal(U[0])) qnan(s.p);
  return s;
}

__device__ __forceinline__ void hllc_x_fp64(const double* UL, const double* UR, double gam,
                                            double* F, double& pL, double& pR) {
  const double gm1 = gam - 1.0;
  const Side L = side_of(UL, gam, gm1), R = side_of(UR, gam, gm1);
  pL = L.p;
  pR = R.p;
  const double SL = min_num(L.u - L.c, R.u - R.c);
  const double SR = max_num(L.u + L.c, R.u + R.c);
  const double dL = SL - L.u, dR = SR - R.u;
  const double qL = __dmul_rn(UL[0], dL), qR = __dmul_rn(UR[0], dR);
  const double num = fma(-R.u, qR, fma(L.u, qL, R.p - L.p));
  const double Ss = __dmul_rn(num, recip_int(qL - qR));
  const bool left = ge0_num(Ss);
  const bool useL = ge0_num(SL);
  const bool useS = left || gt0_num(SR);
  const bool star = !useL && useS;
  // the side the flux is taken on: of the contact, or of the wave that has
  // passed the face
  const bool sideL = useL || (useS && left);
  const double uK = sideL ? L.u : R.u, pK = sideL ? L.p : R.p, EK = sideL ? UL[3] : UR[3];
  const double mK = sideL ? UL[1] : UR[1];
  const double vK = sideL ? L.v : R.v;
  const double SK = sideL ? SL : SR, dK = sideL ? dL : dR, qK = sideL ? qL : qR;
  const double u = star ? Ss : uK;
  const double iD = recip_int(SK - u);
  const double p = fma(qK, u - uK, pK);
  const double H = __dmul_rn(iD, fma(dK, EK, fma(p, SK, -__dmul_rn(pK, uK))));
  const double fs = __dmul_rn(__dmul_rn(qK, iD), u);
  const double f = star ? fs : mK;
  F[0] = f;
  F[1] = fma(f, u, p);
  F[2] = __dmul_rn(f, vK);
  F[3] = __dmul_rn(u, H);
  if (!(L.ok && R.ok)) {
#pragma unroll
    for (int v = 0; v < 4; ++v) qnan(F[v]);
  }
}

__device__ __forceinline__ void hll_x_fp64(const double* UL, const double* UR, double gam,
                                           double* F, double& pL, double& pR) {
  const double gm1 = gam - 1.0;
  const Side L = side_of(UL, gam, gm1), R = side_of(UR, gam, gm1);
  pL = L.p;
  pR = R.p;
  const double SL = min_num(L.u - L.c, R.u - R.c);
  const double SR = max_num(L.u + L.c, R.u + R.c);
  // physical fluxes by the same rounded sequence on both sides
  const double FL[4] = {UL[1], fma(UL[1], L.u, L.p), __dmul_rn(UL[1], L.v),
                        __dmul_rn(L.u, UL[3] + L.p)};
  const double FR[4] = {UR[1], fma(UR[1], R.u, R.p), __dmul_rn(UR[1], R.v),
                        __dmul_rn(R.u, UR[3] + R.p)};
  // F = a F_L - b F_R + c (U_R - U_L), a = S_R / w, b = S_L / w, c = S_L S_R / w,
  // w = S_R - S_L
  const double iw = recip_int(SR - SL);
  const double a = __dmul_rn(SR, iw), b = __dmul_rn(SL, iw), c = __dmul_rn(__dmul_rn(SL, SR), iw);
  const bool useL = ge0_num(SL), useR = !gt0_num(SR);
  const bool dom = L.ok && R.ok;
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    // x-mirror: (L, R, a, b, c) -> (R', L', -b, -a, c) swaps the two products;
    // each is rounded on its own so the mirror face negates exactly
    const double d = __dmul_rn(a, FL[v]) - __dmul_rn(b, FR[v]);
    const double Fm = fma(c, UR[v] - UL[v], d);
    F[v] = useL ? FL[v] : (useR ? FR[v] : Fm);
    if (!dom) qnan(F[v]);
  }
}

// the Riemann solver of the grid (Grid::riemann: 0 HLLC, 1 HLL)
template <class Real>
__device__ __forceinline__ void riemann_x(int kind, const Real* UL, const Real* UR, Real gam,
                                          Real* F, Real& pL, Real& pR) {
  if constexpr (sizeof(Real) == sizeof(double)) {
    if (kind == 1) hll_x_fp64(UL, UR, gam, F, pL, pR);
    else hllc_x_fp64(UL, UR, gam, F, pL, pR);
  } else {
    if (kind == 1) hll_x<Real>(UL, UR, gam, F, pL, pR);
    else hllc_x<Real>(UL, UR, gam, F, pL, pR);
  }
}

// ---------------------------------------------------------------------------
// ghost cells: one kernel over all ghost cells.  The x-ghosts of interior rows
// are set from the W/E rule; the y-ghost rows (corners included) from the S/N
// rule applied to the (possibly x-ghost) cell they copy.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void load_cell(const double* X, const Grid& g, int i, int j,
                                          double* S) {
#pragma unroll
  for (int v = 0; v < 4; ++v) S[v] = X[gidx(g, v, i, j)];
}

// the per-direction CFL rate of one cell, max((|u|+c)/dx, (|v|+c)/dy): the
// admissible step is CFL over its maximum over the cells (the minimum of
// dx/(|u|+c) and dy/(|v|+c), reduced as a maximum of rates so that each cell
// needs one reciprocal and no division).  False: no admissible step (the
// rate NaN, infinite or zero; p / rho < 0 gives NaN).
__device__ __forceinline__ bool cell_rate(const double* S, const Grid& g, double& rate) {
  const double ir = pos_normal(S[0]) ? recip_int(S[0]) : recip(S[0]);
  const double u = S[1] * ir, v = S[2] * ir;
  const double p = (g.gamma - 1.0) * (S[3] - 0.5 * (S[1] * u + S[2] * v));
  const double z = g.gamma * p * ir;
  const double cs = pos_normal(z) ? sqrt_int(z) : sqrt(z);
  const double ax = (fabs(u) + cs) * g.inv_dx, ay = (fabs(v) + cs) * g.inv_dy;
  rate = (g.dim == 1 || lt_ieee(ay, ax)) ? ax : ay;  // a NaN state makes both rates NaN
  return pos_finite(rate);
}

// the same rate on the FP32 path: from the float shadow, in float
__device__ __forceinline__ bool cell_rate(const float* S, const Grid& g, double& rate) {
  const float gam = (float)g.gamma;
  const float ir = recip(S[0]);
  const float u = S[1] * ir, v = S[2] * ir;
  const float p = (gam - 1.0f) * (S[3] - 0.5f * (S[1] * u + S[2] * v));
  const float cs = sqrt_r(gam * p * ir);
  const float ax = (fabsf(u) + cs) * (float)g.inv_dx, ay = (fabsf(v) + cs) * (float)g.inv_dy;
  const float r = (g.dim == 1 || ax > ay) ? ax : ay;
  rate = (double)r;
  return r > 0.0f && isfinite(r);
}

// the rate of cell (i, j): the double state, or its float shadow when Xf is set
__device__ __forceinline__ bool cell_rate_at(const double* X, const float* Xf, const Grid& g,
                                             int i, int j, double& rate) {
  if (Xf) {
    float S[4];
#pragma unroll
    for (int v = 0; v < 4; ++v) S[v] = Xf[gidx(g, v, i, j)];
    return cell_rate(S, g, rate);
  }
  double S[4];
  load_cell(X, g, i, j, S);
  return cell_rate(S, g, rate);
}

// value of the x-ghost (i outside [0,nx)) of interior row j
__device__ __forceinline__ void xghost(const double* X, const Grid& g, int i, int j, double* S) {
  int side = i < 0 ? 0 : 1;
  int k = i < 0 ? -i : i - g.nx + 1;  // ghost layer 1..H
  int kind = g.bc[side];
  if (kind == 3) {
#pragma unroll
    for (int v = 0; v < 4; ++v) S[v] = g.bcU[side][v];
    return;
  }
  int src;
  if (kind == 0) src = wrapi(i, g.nx);
  else if (kind == 2) src = side == 0 ? k - 1 : g.nx - k;
  else src = side == 0 ? 0 : g.nx - 1;
  load_cell(X, g, src, j, S);
  if (kind == 2) S[1] = -S[1];
}

__device__ __forceinline__ void column_cell(const double* X, const Grid& g, int i, int j,
                                            double* S) {
  if (i < 0 || i >= g.nx) xghost(X, g, i, j, S);
  else load_cell(X, g, i, j, S);
}

// ghost cell number tid of the grid (x-ghosts of interior rows first, then
// the ghost rows, corners included), at time t; tid beyond the ghost count
// does nothing
__device__ __forceinline__ long long ghost_count(const Grid& g) {
  return (long long)g.ny * 2 * g.H + (long long)2 * g.H * (g.nx + 2 * g.H);
}

// Xf: the float shadow of X (FP32 path), filled alongside, or null
__device__ __forceinline__ void fill_ghost(double* X, float* Xf, const Grid& g, double t,
                                           long long tid) {
  const int H = g.H;
  const int nxg = g.nx + 2 * H;
  const long long nxs = (long long)g.ny * 2 * H;  // x-ghosts of interior rows
  const long long nys = (long long)2 * H * nxg;   // y-ghost rows
  if (tid >= nxs + nys) return;
  double S[4];
  int i, j;
  if (tid < nxs) {
    j = (int)(tid / (2 * H));
    int c = (int)(tid % (2 * H));
    i = c < H ? -1 - c : g.nx + (c - H);
    xghost(X, g, i, j, S);
  } else {
    long long u = tid - nxs;
    int r = (int)(u / nxg);
    i = (int)(u % nxg) - H;
    int side = r < H ? 0 : 1;  // 0: south, 1: north
    int k = r < H ? r + 1 : r - H + 1;
    j = side == 0 ? -k : g.ny - 1 + k;
    int kind = g.bc[2 + side];
    double xc = g.x0 + (i + 0.5) * g.dx;
    bool fixed = false, reflect = false;
    const double* P = nullptr;
    if (kind == 3) {
      fixed = true;
      P = g.bcU[2 + side];
    } else if (kind == 4) {
      if (xc < g.dmr_wall_x0) {
        fixed = true;
        P = g.dmr_post;
      } else {
        reflect = true;
      }
    } else if (kind == 5) {
      fixed = true;
      P = (xc < g.dmr_xs0 + g.dmr_xs_speed * t) ? g.dmr_post : g.dmr_pre;
    } else if (kind == 6) {
      // jet inflow inside the slit (cell centres), outflow elsewhere
      if (xc >= g.jet_x0 && xc <= g.jet_x1) {
        fixed = true;
        P = g.jetU[side];
      }
    } else if (kind == 2) {
      reflect = true;
    }
    if (fixed) {
#pragma unroll
      for (int v = 0; v < 4; ++v) S[v] = P[v];
    } else {
      int src;
      if (kind == 0) src = wrapi(j, g.ny);
      else if (reflect) src = side == 0 ? k - 1 : g.ny - k;
      else src = side == 0 ? 0 : g.ny - 1;
      column_cell(X, g, i, src, S);
      if (reflect) S[2] = -S[2];
    }
  }
#pragma unroll
  for (int v = 0; v < 4; ++v) X[gidx(g, v, i, j)] = S[v];
  if (Xf) {
#pragma unroll
    for (int v = 0; v < 4; ++v) Xf[gidx(g, v, i, j)] = (float)S[v];
  }
}

// Real copy of a ghosted state: the float shadow of the FP32 path (and of
// the FP32 adjoint), Y = (Real)X elementwise
template <class Real>
__global__ void k_to_real(const double* X, Real* Y, long long n) {
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n;
       t += (long long)gridDim.x * blockDim.x)
    Y[t] = (Real)X[t];
}

// ---------------------------------------------------------------------------
// face-state check of cell (i, j): a state that its own stencil produced on
// one of its four faces, at the face's current radius, failed (non-finite or
// non-positive density or pressure).  Periodic seams need no care: a seam
// face's state of the cell across the seam is computed from the same data at
// the cell's own face; other ghosts' states flag nothing.
// ---------------------------------------------------------------------------
template <class Real>
__device__ __forceinline__ bool face_state_bad(const StageArgs<Real>& A, const Grid& g, int i,
                                               int j) {
  const long long wf = (long long)j * (g.nx + 1) + i;  // x face i: W face of (i, j)
  int b = (A.fbx[wf] >> 1) | A.fbx[wf + 1];            // its right / the E face's left state
  if (g.dim == 2) {
    const long long sf = (long long)j * g.nx + i;       // y face j: S face of (i, j)
    b |= (A.fby[sf] >> 1) | A.fby[sf + g.nx];
  }
  return (b & 1) != 0;
}

// ---------------------------------------------------------------------------
// the face-state tape of a recorded step (Control::stape): the states the
// step's final fluxes were solved from, so that the adjoint need not
// reconstruct them again.  Per stage: x faces (left, right states), y faces
// (lower, upper), each [4 variables][qt points][faces of that direction],
// qt the rule size of the top radius.  Null when the step records none.
// ---------------------------------------------------------------------------
template <class Real>
__device__ __forceinline__ Real* state_tape(const StageArgs<Real>& A, const Grid& g, int qt,
                                            int dir, int side) {
  Real* base = (Real*)A.sc->ctl.stape;
  if (!base) return nullptr;
  const long long nfx = (long long)(g.nx + 1) * g.ny, nfy = (long long)g.nx * (g.ny + 1);
  base += (long long)A.stage * 8 * qt * (nfx + nfy);
  return dir == 0 ? base + (long long)side * 4 * qt * nfx
                  : base + 8LL * qt * nfx + (long long)side * 4 * qt * nfy;
}

// the states UL / UR of point q of face f (of its direction) into the tape
template <class Real>
__device__ __forceinline__ void tape_states(Real* tL, Real* tR, int qt, long long nf, long long f,
                                            int q, const Real* UL, const Real* UR) {
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    tL[((long long)v * qt + q) * nf + f] = UL[v];
    tR[((long long)v * qt + q) * nf + f] = UR[v];
  }
}

// the same for the face between (iL, jL) and its neighbour in direction DIR
// (a periodic seam face: both copies), when the step records states
template <class Real, int DIR>
__device__ __forceinline__ void tape_face(const StageArgs<Real>& A, const Grid& g, int qt, int iL,
                                          int jL, int q, const Real* UL, const Real* UR) {
  Real* tL = state_tape<Real>(A, g, qt, DIR, 0);
  if (!tL) return;
  Real* tR = state_tape<Real>(A, g, qt, DIR, 1);
  if (DIR == 0) {
    const long long nf = (long long)(g.nx + 1) * g.ny;
    const int f = iL + 1;
    tape_states(tL, tR, qt, nf, (long long)jL * (g.nx + 1) + f, q, UL, UR);
    if (g.periodic_x && (f == 0 || f == g.nx))
      tape_states(tL, tR, qt, nf, (long long)jL * (g.nx + 1) + (f == 0 ? g.nx : 0), q, UL, UR);
  } else {
    const long long nf = (long long)g.nx * (g.ny + 1);
    const int f = jL + 1;
    tape_states(tL, tR, qt, nf, (long long)f * g.nx + iL, q, UL, UR);
    if (g.periodic_y && (f == 0 || f == g.ny))
      tape_states(tL, tR, qt, nf, (long long)(f == 0 ? g.ny : 0) * g.nx + iL, q, UL, UR);
  }
}

// ---------------------------------------------------------------------------
// first-pass faces at the top radius R.  One warp covers 32 consecutive
// cells of a row (x_faces) or a column (y_faces) and produces the 31 faces
// between them; the left/lower states come from the neighbouring lane.
// ---------------------------------------------------------------------------
// shared-memory tile of one face block: the block's cells and their
// stencils, converted to Real once, as tile[v][across][along]: "along" runs
// with the sweep (the lanes), "across" with the warps, so every stencil read
// of a warp is one contiguous row of shared memory
template <int R, class Real, int FW>
struct FaceTile {
  static constexpr int TF = kSegCells + 2 * R;
  static constexpr int TS = FW + 2 * R;
  Real t[4][TS][TF];
};

// stage the ghosted state X (any element type) around the block whose first
// cell is `first_fast` along the sweep and `first_slow` across it into the
// shared tile, as Real
template <int R, class Real, int DIR, int FW, class TX>
__device__ __forceinline__ void tile_load_at(FaceTile<R, Real, FW>& T_, const TX* X,
                                             const Grid& g, int first_fast, int first_slow) {
  constexpr int TF = FaceTile<R, Real, FW>::TF;
  constexpr int TS = FaceTile<R, Real, FW>::TS;
  constexpr int NE = TS * TF;                 // tile cells of one variable
  constexpr int NT = 32 * FW;                 // threads of the block
  constexpr int NP = (NE + NT - 1) / NT;      // tile cells per thread
  Real* tile = &T_.t[0][0][0];
  const int tid = threadIdx.y * 32 + threadIdx.x;
  const int fast0 = first_fast - R;           // first tile cell along the sweep
  const int slow0 = first_slow - R;           // first tile cell across it
  // the cells this thread stages, worked out once for the four variables:
  // consecutive threads take consecutive cells along x (coalesced loads)
  long long off[NP];
  int soff[NP];
  bool ok[NP];
#pragma unroll
  for (int p = 0; p < NP; ++p) {
    const int r = tid + p * NT;
    int sl, fa;
    if (DIR == 0) { sl = r / TF; fa = r - sl * TF; }
    else { fa = r / TS; sl = r - fa * TS; }
    const int i = DIR == 0 ? fast0 + fa : slow0 + sl;
    const int j = DIR == 0 ? slow0 + sl : fast0 + fa;
    ok[p] = i >= -g.H && i < g.nx + g.H && j >= -g.H && j < g.ny + g.H;
    off[p] = gidx(g, 0, i, j);  // dereferenced only when ok
    soff[p] = sl * TF + fa;
  }
#pragma unroll
  for (int v = 0; v < 4; ++v)
#pragma unroll
    for (int p = 0; p < NP; ++p)
      if (tid + p * NT < NE)
        tile[v * NE + soff[p]] = ok[p] ? (Real)__ldg(X + off[p] + v * g.vstride) : Real(0);
}

// the tile of segment `seg` along the sweep and band `band` across it
template <int R, class Real, int DIR, int FW, class TX>
__device__ __forceinline__ void tile_load(FaceTile<R, Real, FW>& T_, const TX* X, const Grid& g,
                                          int seg, int band) {
  tile_load_at<R, Real, DIR, FW>(T_, X, g, seg * kSegFaces - 1, band * FW);
}

// states at all Gauss points of the two faces of one tile cell across the
// sweep (top radius R): SP on the +1/2 side (east / north), SM on the -1/2
// side (west / south).  (fl, sw): the cell's tile position along / across.
template <int R, class Real, int DIR, int FW>
__device__ __forceinline__ void tile_face_states(const FaceTile<R, Real, FW>& T_,
                                                 const ParityW<Real>& W, int fl, int sw,
                                                 bool live, Real (&SP)[rule_q(R)][4],
                                                 Real (&SM)[rule_q(R)][4]) {
  constexpr int Q = rule_q(R);
  constexpr int NS = (Q + 1) / 2;
  auto& tile = T_.t;
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    // (a, b): offsets along x and y
    auto ld = [&](int a, int b) -> Real {
      return DIR == 0 ? tile[v][sw + b][fl + a] : tile[v][sw + a][fl + b];
    };
    Recon<R, Real> rc;
    rc.sums(ld, live);
#pragma unroll
    for (int kk = 0; kk < NS; ++kk) {
      typename Recon<R, Real>::T T[2][2];
      rc.dot(DIR == 0 ? W.cx[kk] : W.cy[kk], T);
      const bool middle = (Q & 1) && kk == Q / 2;
      // DIR 0: e even, o odd along x (east / west); DIR 1: along y (north / south)
      const auto t01 = DIR == 0 ? T[0][1] : T[1][0], t10 = DIR == 0 ? T[1][0] : T[0][1];
      if (middle) {
        SP[kk][v] = rc.out(T[0][0] + t10, W);
        SM[kk][v] = rc.out(T[0][0] - t10, W);
      } else {
        const auto e = T[0][0] + t01, o = t10 + T[1][1];
        const auto e2 = T[0][0] - t01, o2 = t10 - T[1][1];
        SP[kk][v] = rc.out(e + o, W);            // E or N (+g)
        SM[kk][v] = rc.out(e - o, W);            // W or S (+g)
        SP[Q - 1 - kk][v] = rc.out(e2 + o2, W);  // E or N (-g)
        SM[Q - 1 - kk][v] = rc.out(e2 - o2, W);  // W or S (-g)
      }
    }
  }
}

// one block of the first-pass face sweep (DIR 0: x faces, 1: y faces) over
// segment `seg` along the sweep and band `band` of FW rows/columns across it
template <int R, class Real, int DIR, int FW>
__device__ __forceinline__ void faces_block(const StageArgs<Real>& A, const Grid& g,
                                            const ParityW<Real>& W, int seg, int band,
                                            FaceTile<R, Real, FW>& T_) {
  constexpr int Q = rule_q(R);
  tile_load<R, Real, DIR, FW>(T_, A.Xr, g, seg, band);
  __syncthreads();
  const int lane = threadIdx.x, warp = threadIdx.y;
  // DIR 0: lanes along x, warp per row; DIR 1: lanes along y, warp per column
  int i, j, nlen, across;
  if (DIR == 0) {
    j = band * FW + warp;
    i = seg * kSegFaces - 1 + lane;
    nlen = g.nx;
    across = g.ny;
  } else {
    i = band * FW + warp;
    j = seg * kSegFaces - 1 + lane;
    nlen = g.ny;
    across = g.nx;
  }
  if ((DIR == 0 ? j : i) >= across) return;  // whole warp
  const int pos = DIR == 0 ? i : j;  // position along the sweep, -1 .. nlen
  const bool live = pos <= nlen;
  Real SP[Q][4], SM[Q][4];
  tile_face_states<R, Real, DIR, FW>(T_, W, lane + R, warp + R, live, SP, SM);
  // left/lower state of the face between this cell and the previous one
  Real SL[Q][4];
#pragma unroll
  for (int q = 0; q < Q; ++q)
#pragma unroll
    for (int v = 0; v < 4; ++v) SL[q][v] = __shfl_up_sync(0xffffffffu, SP[q][v], 1);
  // face index = pos (between pos-1 and pos)
  if (lane == 0 || pos < 0 || pos > nlen) return;
  const Real gam = (Real)g.gamma;
  Real F[4] = {0, 0, 0, 0};
  bool badL = false, badR = false;
  auto point = [&](int q, Real* f) {
    Real pl, pr;
    if (DIR == 0) {
      riemann_x<Real>(g.riemann, SL[q], SM[q], gam, f, pl, pr);
    } else {
      Real a[4] = {SL[q][0], SL[q][2], SL[q][1], SL[q][3]};
      Real b[4] = {SM[q][0], SM[q][2], SM[q][1], SM[q][3]};
      Real h[4];
      riemann_x<Real>(g.riemann, a, b, gam, h, pl, pr);
      f[0] = h[0]; f[1] = h[2]; f[2] = h[1]; f[3] = h[3];
    }
    // face-state check: finite and positive density and pressure (the
    // solver's sound speed needs gamma p / rho > 0; NaN fails the test)
    badL |= !(pos_finite(SL[q][0]) && pos_finite(pl));
    badR |= !(pos_finite(SM[q][0]) && pos_finite(pr));
  };
  // the Gauss points in mirror pairs (g, -g), each pair summed first: a
  // mirror image of the problem that reverses the points sums alike
#pragma unroll
  for (int kk = 0; kk < (Q + 1) / 2; ++kk) {
    Real f1[4];
    point(kk, f1);
    if (Q - 1 - kk != kk) {
      Real f2[4];
      point(Q - 1 - kk, f2);
#pragma unroll
      for (int v = 0; v < 4; ++v) F[v] = fma(W.w[kk], add_rn(f1[v], f2[v]), F[v]);
    } else {
#pragma unroll
      for (int v = 0; v < 4; ++v) F[v] = fma(W.w[kk], f1[v], F[v]);
    }
  }
  if (DIR == 0) {
#pragma unroll
    for (int v = 0; v < 4; ++v) A.Fx[fxidx(g, v, i, j)] = F[v];
    A.fbx[(long long)j * (g.nx + 1) + i] = (uint8_t)((badL ? 1 : 0) | (badR ? 2 : 0));
  } else {
#pragma unroll
    for (int v = 0; v < 4; ++v) A.Fy[fyidx(g, v, i, j)] = F[v];
    A.fby[(long long)j * g.nx + i] = (uint8_t)((badL ? 1 : 0) | (badR ? 2 : 0));
  }
  // a recorded step keeps the states for its adjoint
  if (Real* tL = state_tape<Real>(A, g, Q, DIR, 0)) {
    Real* tR = state_tape<Real>(A, g, Q, DIR, 1);
    const long long nf = DIR == 0 ? (long long)(g.nx + 1) * g.ny : (long long)g.nx * (g.ny + 1);
    const long long f = DIR == 0 ? (long long)j * (g.nx + 1) + i : (long long)j * g.nx + i;
#pragma unroll
    for (int q = 0; q < Q; ++q) tape_states(tL, tR, Q, nf, f, q, SL[q], SM[q]);
  }
}

template <int R, class Real, int DIR, int FW>
__global__ void __launch_bounds__(32 * FW) k_faces(StageArgs<Real> A, Grid g,
                                                   const __grid_constant__ ParityW<Real> W) {
  pdl_wait();
  pdl_trigger();
  __shared__ FaceTile<R, Real, FW> tile;
  faces_block<R, Real, DIR, FW>(A, g, W, DIR == 0 ? blockIdx.x : blockIdx.y,
                                DIR == 0 ? blockIdx.y : blockIdx.x, tile);
}

// ---------------------------------------------------------------------------
// both first-pass face sweeps in one block (two-dimensional grids, FP32).
// Bound by issue (76%; FMA and ALU pipes 38% each): 0.35 ms a launch at
// 4096 x 1024, R = 3, 2200 instructions a warp, half of them in the eight
// Riemann solves.  A block of 8 warps covers 8 rows of a 32-cell segment: lane l, warp w hold cell
// (i0 + l, j0 + w), i0 = 31 seg - 1, j0 = 7 band - 1, so segments overlap by
// one column and bands by one row.  Each cell forms its parity sums once per
// variable and from them both its x states (E/W, kept in registers for the
// x faces, taken from the neighbouring lane by shuffle) and its y states
// (N/S, written to shared memory for the y faces between consecutive rows).
// A thread with l, w >= 1 then solves the x face between (i-1, j) and
// (i, j) and the y face between (i, j-1) and (i, j).  The arithmetic of
// every state and flux is that of the separate sweeps (k_faces), so the
// fluxes are the same bit for bit; y fluxes are stored with lanes along x.
// ---------------------------------------------------------------------------
constexpr int kXYRows = 8;               // cell rows of a fused face block (its warps)
constexpr int kXYBand = kXYRows - 1;     // face rows a block owns

template <int R, class Real>
struct XYShared {
  FaceTile<R, Real, kXYRows> tile;
  Real ys[2][rule_q(R)][4][kXYRows][32];  // [N, S][point][variable][row][lane]
};

// one fused block: segment `seg` (31 x faces) and band `band` (7 rows of
// faces) of the grid
template <int R, class Real>
__device__ __forceinline__ void faces_xy_block(const StageArgs<Real>& A, const Grid& g,
                                               const ParityW<Real>& W, int seg, int band,
                                               XYShared<R, Real>& S) {
  constexpr int Q = rule_q(R);
  constexpr int NS = (Q + 1) / 2;
  const int lane = threadIdx.x, warp = threadIdx.y;
  const int i0 = seg * kSegFaces - 1, j0 = band * kXYBand - 1;
  tile_load_at<R, Real, 0, kXYRows>(S.tile, A.Xr, g, i0, j0);
  __syncthreads();
  const int i = i0 + lane, j = j0 + warp;
  // rows beyond the last y face take no part (their states feed nothing)
  const bool row_live = j <= g.ny;
  const bool xrow = warp >= 1 && j < g.ny;  // this warp's x faces are the block's
  Real SP[Q][4], SM[Q][4];
  auto& tile = S.tile.t;
  const int fl = lane + R, sw = warp + R;
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    auto ld = [&](int a, int b) -> Real { return tile[v][sw + b][fl + a]; };
    Recon<R, Real> rc;
    rc.sums(ld, row_live);
#pragma unroll
    for (int kk = 0; kk < NS; ++kk) {
      const bool middle = (Q & 1) && kk == Q / 2;
      typename Recon<R, Real>::T T[2][2];
      if (xrow) {
        // east / west at +g and -g (the x sweep's butterflies)
        rc.dot(W.cx[kk], T);
        if (middle) {
          SP[kk][v] = rc.out(T[0][0] + T[1][0], W);
          SM[kk][v] = rc.out(T[0][0] - T[1][0], W);
        } else {
          const auto e = T[0][0] + T[0][1], o = T[1][0] + T[1][1];
          const auto e2 = T[0][0] - T[0][1], o2 = T[1][0] - T[1][1];
          SP[kk][v] = rc.out(e + o, W);
          SM[kk][v] = rc.out(e - o, W);
          SP[Q - 1 - kk][v] = rc.out(e2 + o2, W);
          SM[Q - 1 - kk][v] = rc.out(e2 - o2, W);
        }
      }
      // north / south at +g and -g (the y sweep's butterflies), to shared memory
      rc.dot(W.cy[kk], T);
      if (middle) {
        S.ys[0][kk][v][warp][lane] = rc.out(T[0][0] + T[0][1], W);
        S.ys[1][kk][v][warp][lane] = rc.out(T[0][0] - T[0][1], W);
      } else {
        const auto e = T[0][0] + T[1][0], o = T[0][1] + T[1][1];
        const auto e2 = T[0][0] - T[1][0], o2 = T[0][1] - T[1][1];
        S.ys[0][kk][v][warp][lane] = rc.out(e + o, W);
        S.ys[1][kk][v][warp][lane] = rc.out(e - o, W);
        S.ys[0][Q - 1 - kk][v][warp][lane] = rc.out(e2 + o2, W);
        S.ys[1][Q - 1 - kk][v][warp][lane] = rc.out(e2 - o2, W);
      }
    }
  }
  const Real gam = (Real)g.gamma;
  // x faces: the left state from the neighbouring lane
  if (xrow) {
    Real SL[Q][4];
#pragma unroll
    for (int q = 0; q < Q; ++q)
#pragma unroll
      for (int v = 0; v < 4; ++v) SL[q][v] = __shfl_up_sync(0xffffffffu, SP[q][v], 1);
    if (lane >= 1 && i <= g.nx) {
      Real F[4] = {0, 0, 0, 0};
      bool badL = false, badR = false;
      auto point = [&](int q, Real* f) {
        Real pl, pr;
        riemann_x<Real>(g.riemann, SL[q], SM[q], gam, f, pl, pr);
        badL |= !(pos_finite(SL[q][0]) && pos_finite(pl));
        badR |= !(pos_finite(SM[q][0]) && pos_finite(pr));
      };
#pragma unroll
      for (int kk = 0; kk < NS; ++kk) {
        Real f1[4];
        point(kk, f1);
        if (Q - 1 - kk != kk) {
          Real f2[4];
          point(Q - 1 - kk, f2);
#pragma unroll
          for (int v = 0; v < 4; ++v) F[v] = fma(W.w[kk], add_rn(f1[v], f2[v]), F[v]);
        } else {
#pragma unroll
          for (int v = 0; v < 4; ++v) F[v] = fma(W.w[kk], f1[v], F[v]);
        }
      }
#pragma unroll
      for (int v = 0; v < 4; ++v) A.Fx[fxidx(g, v, i, j)] = F[v];
      A.fbx[(long long)j * (g.nx + 1) + i] = (uint8_t)((badL ? 1 : 0) | (badR ? 2 : 0));
      if (Real* tL = state_tape<Real>(A, g, Q, 0, 0)) {
        Real* tR = state_tape<Real>(A, g, Q, 0, 1);
        const long long nf = (long long)(g.nx + 1) * g.ny, f = (long long)j * (g.nx + 1) + i;
#pragma unroll
        for (int q = 0; q < Q; ++q) tape_states(tL, tR, Q, nf, f, q, SL[q], SM[q]);
      }
    }
  }
  __syncthreads();
  // y faces: the lower state from the row below, both from shared memory
  if (warp >= 1 && lane >= 1 && i < g.nx && j <= g.ny) {
    Real F[4] = {0, 0, 0, 0};
    bool badL = false, badR = false;
    auto point = [&](int q, Real* f) {
      Real a[4], b[4];
      a[0] = S.ys[0][q][0][warp - 1][lane];
      a[1] = S.ys[0][q][2][warp - 1][lane];
      a[2] = S.ys[0][q][1][warp - 1][lane];
      a[3] = S.ys[0][q][3][warp - 1][lane];
      b[0] = S.ys[1][q][0][warp][lane];
      b[1] = S.ys[1][q][2][warp][lane];
      b[2] = S.ys[1][q][1][warp][lane];
      b[3] = S.ys[1][q][3][warp][lane];
      Real h[4], pl, pr;
      riemann_x<Real>(g.riemann, a, b, gam, h, pl, pr);
      f[0] = h[0]; f[1] = h[2]; f[2] = h[1]; f[3] = h[3];
      badL |= !(pos_finite(a[0]) && pos_finite(pl));
      badR |= !(pos_finite(b[0]) && pos_finite(pr));
    };
#pragma unroll
    for (int kk = 0; kk < NS; ++kk) {
      Real f1[4];
      point(kk, f1);
      if (Q - 1 - kk != kk) {
        Real f2[4];
        point(Q - 1 - kk, f2);
#pragma unroll
        for (int v = 0; v < 4; ++v) F[v] = fma(W.w[kk], add_rn(f1[v], f2[v]), F[v]);
      } else {
#pragma unroll
        for (int v = 0; v < 4; ++v) F[v] = fma(W.w[kk], f1[v], F[v]);
      }
    }
#pragma unroll
    for (int v = 0; v < 4; ++v) A.Fy[fyidx(g, v, i, j)] = F[v];
    A.fby[(long long)j * g.nx + i] = (uint8_t)((badL ? 1 : 0) | (badR ? 2 : 0));
    if (Real* tL = state_tape<Real>(A, g, Q, 1, 0)) {
      Real* tR = state_tape<Real>(A, g, Q, 1, 1);
      const long long nf = (long long)g.nx * (g.ny + 1), f = (long long)j * g.nx + i;
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        Real UL[4], UR[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          UL[v] = S.ys[0][q][v][warp - 1][lane];
          UR[v] = S.ys[1][q][v][warp][lane];
        }
        tape_states(tL, tR, Q, nf, f, q, UL, UR);
      }
    }
  }
}

constexpr int kXYBlocks = 4;  // resident blocks an SM of the fused FP32 face kernel

template <int R, class Real>
__global__ void __launch_bounds__(32 * kXYRows, kXYBlocks) k_faces_xy(StageArgs<Real> A, Grid g,
                                                           const __grid_constant__ ParityW<Real> W) {
  pdl_wait();
  pdl_trigger();
  extern __shared__ __align__(16) unsigned char xy_smem[];
  XYShared<R, Real>& S = *reinterpret_cast<XYShared<R, Real>*>(xy_smem);
  faces_xy_block<R, Real>(A, g, W, blockIdx.x, blockIdx.y, S);
}

// ---------------------------------------------------------------------------
// detection, Steps 4-9 (eqs. CAD, PAD, divV, gradP, plateau, DMP_RK,
// u2_curvature, u2_a, u2_b) on the candidate Y of cell (i,j) with the ghosted
// stage input X.  Returns true for a troubled cell.
// ---------------------------------------------------------------------------
// a detection constant in the precision of the tests (Detect holds both)
template <class Real>
__device__ __forceinline__ Real det_c(double d, float f);
template <>
__device__ __forceinline__ double det_c<double>(double d, float) { return d; }
template <>
__device__ __forceinline__ float det_c<float>(double, float f) { return f; }

// a double in the precision of the tests: FP32 rounds it on the integer pipes
template <class Real>
__device__ __forceinline__ Real to_real(double x);
template <>
__device__ __forceinline__ double to_real<double>(double x) { return x; }
template <>
__device__ __forceinline__ float to_real<float>(double x) { return fpb_double_to_float_rn(x); }

template <class Real>
__device__ __forceinline__ Real xload(const Real* X, const Grid& g, int v, int i, int j) {
  return X[gidx(g, v, i, j)];  // not __ldg: the 1D step kernel has written X itself
}

// What Steps 6, 7 and 9 find depends on the stage input alone, not on the
// candidate, so a cell detected again in the same stage need not repeat it.
// What is known of a cell is kept in bits 2-3 of the byte of its W face:
constexpr int kVerdictNone = 0;    // nothing yet
constexpr int kVerdictAccept = 1;  // accepted by CSD, the plateau or u2
constexpr int kVerdictDmp = 2;     // CSD and plateau failed, u2 not looked at
constexpr int kVerdictDmpOnly = 3; // and u2 failed: accepted by the DMP or not at all
constexpr int kVerdictBits = 12;
constexpr int kVerdictCsdFailed = 4;  // (not kept, see quick_csd)
// (the other bits of the byte change in other phases only)
template <class Real>
__device__ __forceinline__ void keep_verdict(const StageArgs<Real>& A, const Grid& g, int i,
                                             int j, int verdict) {
  uint8_t* b = A.fbx + (long long)j * (g.nx + 1) + i;
  *b = (uint8_t)((*b & ~kVerdictBits) | verdict << 2);
}

// Detection in float, FP64 path, where the float values decide a test whatever
// the rounding.  quick_csd: kVerdictAccept (CAD, PAD and CSD pass),
// kVerdictCsdFailed (CAD and PAD pass, CSD fails) or kVerdictNone (too close
// to a threshold, or CAD or PAD may fail, or out of float's range).  Few cells
// are close, and an FP64 operation costs 64 times a float one: 0.21 ms a launch
// at 4096 x 1024 (the candidate and the RK sums) for 0.78 with the tests in FP64.
// The double -> float cut is below 2^-23 relative and so is every float
// operation on normal numbers; |u|, K = |m|^2 / (2 rho) and E carry at most 8
// such errors, so 2^-19 of their magnitudes bounds each.  Floats lose relative
// accuracy below 2^-126: a momentum cut to zero there moves u by 2^-126 / rho
// (du) and K by nothing, and a square that underflows is off by 2^-149, K by
// 2^-149 / rho, which stays below 2^-28 of E where rho E > 2^-120; elsewhere
// the pressure is not known.  (Detect::quick: the thresholds and mesh widths
// lie within 2^+-60, so that no sum or bound below under- or overflows.)  A NaN
// or an infinity fails every comparison.
struct QuickPrim {
  float w, dw;  // normal velocity and its error bound over 2^-18
  float p, dp;  // pressure / (gamma - 1) and its error bound
};
__device__ __forceinline__ float cut_float(double x) {
  // the leading 24 bits; below the float range zero, beyond it an infinity
  const uint32_t h = fxd_hi(x), l = fxd_lo(x);
  int t = (int)(h & 0x7fffffffu) - (896 << 20);
  t = t < 0 ? 0 : t;
  const uint32_t b = t >= (255 << 20) ? 0x7f800000u : ((uint32_t)t << 3 | (t ? l >> 29 : 0u));
  return __int_as_float((int)(b | (h & 0x80000000u)));
}
__device__ __forceinline__ QuickPrim quick_prim(double r, double mn, double mt, double E) {
  const float rf = cut_float(r), nf = cut_float(mn), tf = cut_float(mt), ef = cut_float(E);
  const float ir = recip(rf);
  const float K = 0.5f * (nf * nf + tf * tf) * ir;
  QuickPrim q;
  q.w = nf * ir;
  q.dw = fmaf(0x1p-106f, ir, fabsf(q.w));
  q.p = rf > 0x1p-100f && rf < 0x1p100f && rf * ef > 0x1p-120f ? ef - K : -1.0f;
  q.dp = 0x1p-19f * (fabsf(ef) + K);
  return q;
}
// CAD and PAD pass
__device__ __forceinline__ bool quick_pad(const double* Y) {
  const QuickPrim y = quick_prim(Y[0], Y[1], Y[2], Y[3]);
  return y.p - y.dp > 0x1p-100f && y.p < 0x1p100f;
}
template <class LX>
__device__ __forceinline__ int quick_csd(const LX& X, const Grid& g, const Detect& D,
                                         const double* Y) {
  if (!D.csd_on || !D.quick) return kVerdictNone;
  bool sure = quick_pad(Y);
  float div = 0.0f, ediv = 0.0f, most = 0.0f, least = 0.0f;  // bounds of the pressure gradient
#pragma unroll
  for (int d = 0; d < 2; ++d) {
    if (d == 1 && g.dim != 2) break;
    const int a = d == 0, b = d == 1;
    const QuickPrim e = quick_prim(X(0, a, b), X(1 + d, a, b), X(2 - d, a, b), X(3, a, b));
    const QuickPrim w = quick_prim(X(0, -a, -b), X(1 + d, -a, -b), X(2 - d, -a, -b), X(3, -a, -b));
    const float h = d == 0 ? D.hx_f : D.hy_f;
    div += (e.w - w.w) * h;
    ediv += (e.dw + w.dw) * h;
    const float low = fminf(e.p - e.dp, w.p - w.dp), high = fminf(e.p + e.dp, w.p + w.dp);
    const float jump = fabsf(e.p - w.p), off = e.dp + w.dp;
    sure = sure && low > 0x1p-100f && high < 0x1p100f;
    most += (jump + off) * recip(low) * h;
    least += fmaxf(jump - off, 0.0f) * recip(high) * h;
  }
  // 2^-18 of the sums of magnitudes covers the errors of the sums too
  const float up = 1.0f + 0x1p-18f, down = 1.0f - 0x1p-18f;
  if (!sure) return kVerdictNone;
  if (div - 0x1p-18f * ediv >= -D.sigma_v_f * down && most * up <= D.sigma_p_f * down)
    return kVerdictAccept;
  if (div + 0x1p-18f * ediv < -D.sigma_v_f * up || least * down > D.sigma_p_f * up)
    return kVerdictCsdFailed;
  return kVerdictNone;
}

// u2: 1 passes, 0 fails, -1 too close.  With S the sum of |w| |rho| of a
// curvature (the largest of the five) a float curvature is within 2^-20.8 S:
// cuts of 2^-23 in both factors, a rounded product, four rounded sums.  What
// underflows, a rho below 2^-126 or a product, moves it by 2^-126 of the sum of
// |w| and by 5 2^-149: nothing next to that where S is above 2^-100 of that sum
// and above 2^-90.
template <class LX>
__device__ __forceinline__ int quick_u2(const LX& X, const Grid& g, const Detect& D,
                                        const double* d2x, const double* d2y) {
  const bool two = g.dim == 2;
  const int ci[5] = {0, -1, 1, 0, 0}, cj[5] = {0, 0, 0, 1, -1};
  const float lowd = D.delta_f * (1.0f - 0x1p-18f), highd = D.delta_f * (1.0f + 0x1p-18f);
  const float up = 1.0f + 0x1p-18f, down = 1.0f - 0x1p-18f;
  if (!D.quick) return -1;
  int pass = 1;
#pragma unroll
  for (int d = 0; d < 2; ++d) {
    if (d == 1 && !two) break;
    float w[5], least = 0x1p-90f;
#pragma unroll
    for (int m = 0; m < 5; ++m) {
      w[m] = cut_float((d == 0 ? d2x : d2y)[m]);
      least = fmaf(0x1p-100f, fabsf(w[m]), least);
    }
    float cmin = 0.0f, cmax = 0.0f, S = 0.0f;
#pragma unroll
    for (int m = 0; m < 5; ++m) {
      if (m >= 3 && !two) break;
      const int a = ci[m], b = cj[m];
      const float t[5] = {w[0] * cut_float(X(0, a, b - 1)), w[1] * cut_float(X(0, a - 1, b)),
                          w[2] * cut_float(X(0, a, b)), w[3] * cut_float(X(0, a + 1, b)),
                          w[4] * cut_float(X(0, a, b + 1))};
      const float k = ((t[0] + t[4]) + (t[1] + t[3])) + t[2];
      S = fmaxf(S, fabsf(t[0]) + fabsf(t[1]) + fabsf(t[2]) + fabsf(t[3]) + fabsf(t[4]));
      cmin = m == 0 ? k : fminf(cmin, k);
      cmax = m == 0 ? k : fmaxf(cmax, k);
    }
    const float e = 0x1p-20f * S;
    if (!(S < 0x1p60f && S > least)) return -1;  // also a NaN
    // the product over the intervals of cmin and cmax
    const float p1 = (cmin - e) * (cmax - e), p2 = (cmin - e) * (cmax + e);
    const float p3 = (cmin + e) * (cmax - e), p4 = (cmin + e) * (cmax + e);
    const float plo = fminf(fminf(p1, p2), fminf(p3, p4)), phi = fmaxf(fmaxf(p1, p2), fmaxf(p3, p4));
    const bool same = plo > 0.0f || -plo < lowd, apart = phi < 0.0f && -phi > highd;
    const float amin = fabsf(cmin), amax = fabsf(cmax), big = fmaxf(amin, amax);
    const bool ua = big + e < lowd, not_ua = big - e > highd;
    const bool ub = amin - e > 0.5f * (amax + e) * up, not_ub = amin + e < 0.5f * (amax - e) * down;
    if (apart || (not_ua && not_ub)) return 0;
    if (!(same && (ua || ub))) pass = -1;
  }
  return pass;
}

// X(v, a, b): variable v of the ghosted stage input at (i + a, j + b), in
// Real; every call below has constant offsets once the loops are unrolled.
// verdict: what is known of the cell (kVerdict*), updated.
template <class Real, class LX>
__device__ __forceinline__ bool troubled_at(const LX& X, const Grid& g, const Detect& D,
                                            const Real* d2x, const Real* d2y, const double* Yd,
                                            int& verdict) {
  const Real gm1 = det_c<Real>(D.gm1, D.gm1_f);
  Real Y[4] = {to_real<Real>(Yd[0]), to_real<Real>(Yd[1]), to_real<Real>(Yd[2]),
               to_real<Real>(Yd[3])};
  Real rho = Y[0];
  bool sure = false, csd_failed = false;  // CAD and PAD passed; CSD failed
  if constexpr (sizeof(Real) == sizeof(double)) {
    if (verdict == kVerdictNone) {
      const int q = quick_csd(X, g, D, Yd);
      if (q == kVerdictAccept) {
        verdict = kVerdictAccept;
        return false;
      }
      sure = csd_failed = q == kVerdictCsdFailed;
    } else {
      sure = quick_pad(Yd);
    }
  }
  if (!sure) {
    Real p = gm1 * (Y[3] - Real(0.5) * (Y[1] * Y[1] + Y[2] * Y[2]) * recip(Y[0]));
    if (!finite_r(rho) || !finite_r(p)) return true;    // Step 4, CAD
    if (!gt0_num(rho) || !gt0_num(p)) return true;       // Step 5, PAD
  }
  if (verdict == kVerdictAccept) return false;
  const bool two = g.dim == 2;  // 1D: the x terms and the W/E neighbours only
  if (verdict == kVerdictNone && !csd_failed && D.csd_on) {  // Step 6, CSD
    Real rE = X(0, 1, 0), rW = X(0, -1, 0);
    Real rN = X(0, 0, 1), rS = X(0, 0, -1);
    Real mxE = X(1, 1, 0), mxW = X(1, -1, 0);
    Real myE = X(2, 1, 0), myW = X(2, -1, 0);
    Real mxN = X(1, 0, 1), mxS = X(1, 0, -1);
    Real myN = X(2, 0, 1), myS = X(2, 0, -1);
    Real eE = X(3, 1, 0), eW = X(3, -1, 0);
    Real eN = X(3, 0, 1), eS = X(3, 0, -1);
    Real iE = recip(rE), iW = recip(rW), iN = recip(rN), iS = recip(rS);
    // one rounded sequence for every neighbour: mirror neighbours agree bitwise
    const Real SE[4] = {rE, mxE, myE, eE}, SW[4] = {rW, mxW, myW, eW};
    const Real SN[4] = {rN, mxN, myN, eN}, SS[4] = {rS, mxS, myS, eS};
    Real uE, uW, vN, vS, tmp;
    Real pE = pressure_ir(SE, iE, gm1, uE, tmp);
    Real pW = pressure_ir(SW, iW, gm1, uW, tmp);
    Real pN = pressure_ir(SN, iN, gm1, tmp, vN);
    Real pS = pressure_ir(SS, iS, gm1, tmp, vS);
    const Real hx = det_c<Real>(D.hx, D.hx_f), hy = det_c<Real>(D.hy, D.hy_f);
    Real mx_ = lt_ieee(pE, pW) ? pE : pW, my_ = lt_ieee(pN, pS) ? pN : pS;
    Real divV = (uE - uW) * hx, gradP = fabs(pE - pW) * hx * recip(mx_);
    if (two) {
      divV += (vN - vS) * hy;
      gradP += fabs(pN - pS) * hy * recip(my_);
    }
    if (le_ieee(-det_c<Real>(D.sigma_v, D.sigma_v_f), divV) &&
        le_ieee(gradP, det_c<Real>(D.sigma_p, D.sigma_p_f))) {
      verdict = kVerdictAccept;
      return false;
    }
  }
  Real r0 = X(0, 0, 0);
  Real rmin = r0, rmax = r0;
  const int di[4] = {-1, 1, 0, 0}, dj[4] = {0, 0, 1, -1};
  const int nnb = two ? 4 : 2;
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    if (m >= nnb) break;
    Real r = X(0, di[m], dj[m]);
    rmin = lt_ieee(r, rmin) ? r : rmin;
    rmax = lt_ieee(rmax, r) ? r : rmax;
  }
  if (verdict == kVerdictNone) {
    if (lt_ieee(rmax - rmin, det_c<Real>(D.plateau_thr, D.plateau_thr_f))) {  // Step 7
      verdict = kVerdictAccept;
      return false;
    }
    verdict = kVerdictDmp;
  }
  if (le_ieee(rmin, rho) && le_ieee(rho, rmax)) return false;     // Step 8, DMP
  if (verdict == kVerdictDmpOnly) return true;
  if constexpr (sizeof(Real) == sizeof(double)) {
    const int q = quick_u2(X, g, D, d2x, d2y);
    if (q >= 0) {
      verdict = q ? kVerdictAccept : kVerdictDmpOnly;
      return q == 0;
    }
  }
  // Step 9, u2 with the App. B second-derivative weights (R=1 stencil in
  // the order b=-1: (0,-1); b=0: (-1,0),(0,0),(1,0); b=1: (0,1))
  const int ci[5] = {0, -1, 1, 0, 0}, cj[5] = {0, 0, 0, 1, -1};
  const Real delta = det_c<Real>(D.delta, D.delta_f);
#pragma unroll
  for (int d = 0; d < 2; ++d) {
    if (d == 1 && !two) break;
    const Real* w = d == 0 ? d2x : d2y;
    Real cmin = Real(0), cmax = Real(0);
#pragma unroll
    for (int m = 0; m < 5; ++m) {
      if (m >= 1 + nnb) break;
      const int a = ci[m], b = cj[m];
      // mirror pairs (S, N) and (W, E) summed first, each product rounded on
      // its own: a mirror-symmetric state gives the same curvature bit for bit
      const Real ks = add_rn(mul_rn(w[0], X(0, a, b - 1)), mul_rn(w[4], X(0, a, b + 1)));
      const Real kw = add_rn(mul_rn(w[1], X(0, a - 1, b)), mul_rn(w[3], X(0, a + 1, b)));
      Real k = add_rn(add_rn(ks, kw), mul_rn(w[2], X(0, a, b)));
      if (m == 0) {
        cmin = k;
        cmax = k;
      } else {
        cmin = lt_ieee(k, cmin) ? k : cmin;
        cmax = lt_ieee(cmax, k) ? k : cmax;
      }
    }
    bool same = lt_ieee(-delta, cmin * cmax);
    Real acmax = fabs(cmax), acmin = fabs(cmin);
    bool ua = same && lt_ieee(lt_ieee(acmin, acmax) ? acmax : acmin, delta);
    // |Cmin|/|Cmax| >= 1/2 written without the division; equal for every
    // non-NaN input once (a) is taken into account
    bool ub = same && le_ieee(Real(0.5) * acmax, acmin);
    if (!(ua || ub)) {
      verdict = kVerdictDmpOnly;
      return true;
    }
  }
  verdict = kVerdictAccept;
  return false;
}

// X: the ghosted stage input in Real; the loads are issued as the tests
// reach them (the first pass: many cells in flight hide their latency)
template <class Real>
__device__ bool troubled(const Real* X, const Grid& g, const Detect& D, const Real* d2x,
                         const Real* d2y, int i, int j, const double* Yd, int& verdict) {
  auto lx = [&](int v, int a, int b) -> Real { return xload<Real>(X, g, v, i + a, j + b); };
  return troubled_at<Real>(lx, g, D, d2x, d2y, Yd, verdict);
}

// candidate of eq. fvm_discrete and the SSP-RK3 combination (eq. rk3) of cell (i,j)
// the stage's flux-difference coefficients h dt / dx and h dt / dy
struct StageC {
  double cx, cy;
};
template <class Real>
__device__ __forceinline__ StageC stage_coeffs(const StageArgs<Real>& A, const Grid& g,
                                               double dt) {
  const double hdt = A.h * dt;
  return StageC{hdt * g.inv_dx, hdt * g.inv_dy};
}

// a load issued where it stands: the MOOD loop's few cells an iteration leave
// every memory latency exposed, and the compiler would move a load that only
// a branch uses into it, behind the loads that decide the branch
__device__ __forceinline__ double load_now(const double* p) {
  double v;
  asm volatile("ld.global.f64 %0, [%1];" : "=d"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ float load_now(const float* p) {
  float v;
  asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ unsigned load_now(const uint8_t* p) {
  unsigned v;
  asm volatile("ld.global.u8 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// 0 or 1 for the trip count of a loop that stands for an if.  FP64 code under an
// if of a few instructions is compiled with predicates, and an FP64 instruction
// no lane takes part in holds the pipe as long as any: the first-pass update
// issued 33 of them a warp in every stage, where the first stage needs 8.
__device__ __forceinline__ int branch(bool cond) {
  int n = cond;
  asm volatile("" : "+r"(n));
  return n;
}
// and x, tied to the loop: what is invariant in it would be formed ahead of it
__device__ __forceinline__ double in_loop(double x) {
  asm volatile("" : "+d"(x));
  return x;
}

// the flux differences fe - fw and gn - gs of NV variables from v0 on, as
// doubles; FP32: on the float and integer pipes (fpb_diff), but for the odd
// cell that is not for it
template <int NV, class Real>
__device__ __forceinline__ void flux_diffs(const StageArgs<Real>& A, const Grid& g, int i, int j,
                                           int v0, double* dx, double* dy) {
  const Real* fx = A.Fx + fxidx(g, v0, i, j);
  const Real* fy = A.Fy + fyidx(g, v0, i, j);
  const long long px = fxidx(g, 1, 0, 0), py = fyidx(g, 1, 0, 0), up = fyidx(g, 0, 0, 1);
  if constexpr (sizeof(Real) == sizeof(float)) {
    bool all = true;
#pragma unroll
    for (int n = 0; n < NV; ++n) {
      int ox, oy;
      dx[n] = fpb_diff(fx[n * px + 1], fx[n * px], &ox);
      dy[n] = fpb_diff(fy[n * py + up], fy[n * py], &oy);
      all = all && ox && oy;
    }
#pragma unroll 1
    for (int t = branch(!all); t > 0; --t)
#pragma unroll
      for (int n = 0; n < NV; ++n) {
        dx[n] = (double)load_now(fx + n * px + 1) - (double)load_now(fx + n * px);
        dy[n] = (double)load_now(fy + n * py + up) - (double)load_now(fy + n * py);
      }
  } else {
#pragma unroll
    for (int n = 0; n < NV; ++n) {
      dx[n] = fx[n * px + 1] - fx[n * px];
      dy[n] = fy[n * py + up] - fy[n * py];
    }
  }
}

// the candidate, NV variables from v0 on
template <int NV, class Real>
__device__ __forceinline__ void candidate(const StageArgs<Real>& A, const Grid& g, int i, int j,
                                          int v0, StageC k, double* Y) {
  double dx[NV], dy[NV];
  flux_diffs<NV, Real>(A, g, i, j, v0, dx, dy);
#pragma unroll
  for (int n = 0; n < NV; ++n)
    Y[n] = fma(-k.cx, dx[n], fma(-k.cy, dy[n], A.X[gidx(g, v0 + n, i, j)]));
}

// the SSP-RK combination of the candidates Y of NV variables, stored at k0 and
// vstride apart: ca u0 + cb Y, with u0 U^n (read where ca is not zero).  The
// first stage's combination is the candidate itself (ca = 0, cb = 1); a cb that
// is a power of two (the second stage's 1/4) only steps exponents.
template <int NV, class Real>
__device__ __forceinline__ void combine(const StageArgs<Real>& A, long long k0, long long vstride,
                                        const double* Y, const double* u0) {
  // compared as integers: an FP64 compare costs what a product does
  const bool with_u0 = __double_as_longlong(A.ca) != 0;
  double o[NV];
#pragma unroll
  for (int n = 0; n < NV; ++n) o[n] = Y[n];
#pragma unroll 1
  for (int t = branch(__double_as_longlong(A.cb) != 0x3ff0000000000000ll); t > 0; --t) {
    const bool pow2 = fpb_is_pow2(A.cb);
    bool product = !pow2;
#pragma unroll
    for (int n = 0; n < NV; ++n) {
      product = product || !fpb_pow2_steps(o[n], A.cb);
      if (pow2) o[n] = fpb_step_exponent(o[n], A.cb);
    }
#pragma unroll 1
    for (int u = branch(product); u > 0; --u)
#pragma unroll
      for (int n = 0; n < NV; ++n) o[n] = A.cb * in_loop(Y[n]);
  }
#pragma unroll 1
  for (int t = branch(with_u0); t > 0; --t)
#pragma unroll
    for (int n = 0; n < NV; ++n) o[n] = fma(A.ca, in_loop(u0[n]), o[n]);
#pragma unroll
  for (int n = 0; n < NV; ++n) {
    A.out[k0 + n * vstride] = o[n];
    if constexpr (sizeof(Real) == sizeof(float))
      A.outr[k0 + n * vstride] = fpb_double_to_float_rn(o[n]);
  }
#pragma unroll 1
  for (int t = branch(A.out2 != nullptr); t > 0; --t)
#pragma unroll
    for (int n = 0; n < NV; ++n)
      A.out2[k0 + n * vstride] = fma(A.wa, A.W[k0 + n * vstride], A.wb * in_loop(Y[n]));
}
template <class Real>
__device__ __forceinline__ void combine_store(const StageArgs<Real>& A, const Grid& g, int i,
                                              int j, const double* Y) {
  double u0[4] = {0.0, 0.0, 0.0, 0.0};
  if (__double_as_longlong(A.ca) != 0) {
#pragma unroll
    for (int v = 0; v < 4; ++v) u0[v] = A.U0[gidx(g, v, i, j)];
  }
  combine<4, Real>(A, gidx(g, 0, i, j), g.vstride, Y, u0);
}

// append to a queue with one atomic per warp
__device__ __forceinline__ void queue_push(bool flag, int cell, int* queue, int* count) {
  unsigned act = __activemask();
  unsigned m = __ballot_sync(act, flag);
  if (m == 0) return;
  int lane = threadIdx.x & 31;
  int leader = __ffs(m) - 1;
  int base = 0;
  if (lane == leader) base = atomicAdd(count, __popc(m));
  base = __shfl_sync(act, base, leader);
  if (flag) queue[base + __popc(m & ((1u << lane) - 1u))] = cell;
}

// first-pass update of cell (i,j) (if in range): candidate, detection,
// RK combination; troubled cells go to the queue as cell_off + local index.
// D and d2x/d2y are the detection constants and App. B weights of the grid.
template <class Real>
__device__ __forceinline__ void update_cell_w(const StageArgs<Real>& A, const Grid& g,
                                              const Detect& D, const DirectW<Real>& Wd,
                                              const Real* d2x, const Real* d2y, int i, int j,
                                              int cell_off, StageC k) {
  const bool in = i < g.nx && j < g.ny;
  bool bad = false;
  int c = 0;
  if (in) {
    c = cidx(g, i, j);
    double Y[4];
    candidate<4, Real>(A, g, i, j, 0, k, Y);
    const int top = Wd.top;
    if (top != 0) {
      int verdict = kVerdictNone;
      bad = face_state_bad<Real>(A, g, i, j) ||
            troubled<Real>(A.Xr, g, D, d2x, d2y, i, j, Y, verdict);
      if (verdict != kVerdictNone) keep_verdict<Real>(A, g, i, j, verdict);
    } else {
      Real y[4] = {(Real)Y[0], (Real)Y[1], (Real)Y[2], (Real)Y[3]};
      Real p = (Real)(g.gamma - 1.0) * (y[3] - Real(0.5) * (y[1] * y[1] + y[2] * y[2]) / y[0]);
      if (!(y[0] > Real(0)) || !(p > Real(0))) atomicAdd(&A.scw->nfog_pad[A.stage], 1);
    }
    A.ord[c] = (uint8_t)top;
    A.first[c] = (uint8_t)bad;
    combine_store<Real>(A, g, i, j, Y);
  }
  queue_push(bad, cell_off + c, A.queue, A.qcount);
}

// FP32 at 4096 x 1024: 0.18 ms a launch, bound by issue (60%) and latency; 0.26
// when it was bound by the FP64 pipe, 33 instructions a warp, of which it needs
// 8 to 16 (see flux_diffs, combine, branch; fp_bits.h on folded compares).  FP64:
// 0.22 ms.  Resident blocks an SM: of 3 to 6 the fastest at this size that is
// not slower on small grids.
template <class Real>
__global__ void __launch_bounds__(256, sizeof(Real) == sizeof(double) ? 4 : 5) k_update_first(StageArgs<Real> A, Grid g, Detect D,
                                                      const __grid_constant__ DirectW<Real> Wd) {
  pdl_wait();
  pdl_trigger();
  // the stage coefficients once per block: FP64 work is charged per warp
  // instruction, so a value every warp computed would cost every warp
  __shared__ StageC k;
  if (threadIdx.x == 0 && threadIdx.y == 0) k = stage_coeffs<Real>(A, g, A.sc->dt);
  __syncthreads();
  update_cell_w<Real>(A, g, D, Wd, Wd.d2x, Wd.d2y, blockIdx.x * blockDim.x + threadIdx.x,
                      blockIdx.y * blockDim.y + threadIdx.y, 0, k);
}

// ---------------------------------------------------------------------------
// MOOD iteration kernels
// ---------------------------------------------------------------------------
// neighbour of (i,j) in direction d (0 W, 1 E, 2 S, 3 N) with periodic wrap;
// returns -1 beyond a non-periodic boundary
__device__ __forceinline__ int neighbour(const Grid& g, int i, int j, int d) {
  int a = i + (d == 0 ? -1 : d == 1 ? 1 : 0);
  int b = j + (d == 2 ? -1 : d == 3 ? 1 : 0);
  if (a < 0 || a >= g.nx) {
    if (!g.periodic_x) return -1;
    a = wrapi(a, g.nx);
  }
  if (b < 0 || b >= g.ny) {
    if (!g.periodic_y) return -1;
    b = wrapi(b, g.ny);
  }
  return cidx(g, a, b);
}

// radius of a possibly-ghost cell now and before this iteration's lowering
__device__ __forceinline__ void radius_pair(const Grid& g, const uint8_t* ord, const uint32_t* stamp,
                                            uint32_t cur, const Cascade& C, int i, int j,
                                            int& now, int& before) {
  const int top = C.top;
  if (i < 0 || i >= g.nx) {
    if (!g.periodic_x) { now = before = top; return; }
    i = wrapi(i, g.nx);
  }
  if (j < 0 || j >= g.ny) {
    if (!g.periodic_y) { now = before = top; return; }
    j = wrapi(j, g.ny);
  }
  int c = cidx(g, i, j);
  now = ord[c];
  before = stamp[c] == cur ? C.prev[now] : now;
}

// one variable of a face state by the direct weights at a radius K <= KM
// given at run time, in fixed point (fixed_dot.h): X points at the cell, z at
// the weights in the slots of the radius-3 diamond.  All loads are issued
// before the first use.
template <int KM>
__device__ __forceinline__ double fx_value(const double* X, int pitch, const int2* z, int K,
                                           int off) {
  double x[stencil_n(KM)];
  int k = 0;
#pragma unroll
  for (int b = -KM; b <= KM; ++b)
#pragma unroll
    for (int a = -KM; a <= KM; ++a) {
      const int ab = (a < 0 ? -a : a) + (b < 0 ? -b : b);
      if (ab <= KM) x[k++] = ab <= K ? X[(long long)b * pitch + a] : 0.0;
    }
  uint32_t top = (uint32_t)FXD_EMIN << 20;
#pragma unroll
  for (int m = 0; m < stencil_n(KM); ++m) top = max(top, fxd_hi(x[m]) & 0x7fffffffu);
  const int E = (int)(top >> 20);
  fxd_acc acc = {0, 0, 0};
  k = 0;
#pragma unroll
  for (int b = -KM; b <= KM; ++b)
#pragma unroll
    for (int a = -KM; a <= KM; ++a)
      if ((a < 0 ? -a : a) + (b < 0 ? -b : b) <= KM) {
        const int2 w = z[diamond3_slot(a, b)];
        const long long v = fxd_from_double(x[k++], E);
        fxd_mac(&acc, w.x, w.y, fxd_limb_hi(v), fxd_limb_lo(v));
      }
  return fxd_to_double(fxd_round(acc), E, off, E == 0x7ff ? 0x7ff80000u : 0u);
}
// out of line: the replay and reverse kernels call it for every variable of
// every state
static __device__ __noinline__ double fx_value_any(const double* X, int pitch, const int2* z,
                                                   int K, int off) {
  return fx_value<3>(X, pitch, z, K, off);
}

// direct reconstruction of one face state at radius K (eq.
// gp_reconstructor): Gauss point q of face 0 E, 1 W, 2 N, 3 S of cell (i, j)
template <int K, class Real>
__device__ __forceinline__ void recon_direct(const Real* X, const Grid& g,
                                             const DirectW<Real>& Wd, int face, int q, int i,
                                             int j, Real* S) {
  const Real* Xc = X + (long long)(j + g.H) * g.pitch + (i + g.H);
  if constexpr (sizeof(Real) == sizeof(double)) {
#pragma unroll
    for (int v = 0; v < 4; ++v)
      S[v] = fx_value_any(Xc + v * g.vstride, g.pitch, Wd.z[K][face][q], K, Wd.off);
  } else {
    // row by row, each row from its centre out in x-mirror pairs (a, -a) with
    // every product rounded on its own: the x-mirror image of the problem,
    // whose weights are the mirrored ones, gives the mirrored state bit for bit
    const Real* z = Wd.z[K][face][q];
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const Real* Xv = Xc + (long long)v * g.vstride;
      Real s = Real(0);
      int row = 0;  // stencil index of the row's first cell
#pragma unroll
      for (int b = -K; b <= K; ++b) {
        const int hb = K - (b < 0 ? -b : b);
        const int mid = row + hb;  // (0, b)
        const Real* Xr = Xv + (long long)b * g.pitch;
        Real t = mul_rn(z[mid], __ldg(Xr));
#pragma unroll
        for (int a = 1; a <= hb; ++a)
          t = add_rn(t, add_rn(mul_rn(z[mid + a], __ldg(Xr + a)), mul_rn(z[mid - a], __ldg(Xr - a))));
        s = add_rn(s, t);
        row += 2 * hb + 1;
      }
      S[v] = s;
    }
  }
}

// Riemann flux at Gauss point q of the face between cell (iL,jL) and its
// neighbour (iR,jR) in direction DIR at radius K; badL / badR gather the
// face-state check of the two reconstructed states
template <int K, class Real, int DIR>
__device__ __forceinline__ void face_point(const Real* X, const Grid& g, const DirectW<Real>& Wd,
                                           int iL, int jL, int q, Real* f, bool& badL,
                                           bool& badR, Real* sUL = nullptr,
                                           Real* sUR = nullptr) {
  const int iR = iL + (DIR == 0), jR = jL + (DIR == 1);
  const Real gam = (Real)g.gamma;
  Real UL[4], UR[4];
  if (K == 0) {
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      UL[v] = __ldg(X + gidx(g, v, iL, jL));
      UR[v] = __ldg(X + gidx(g, v, iR, jR));
    }
  } else {
    recon_direct<K, Real>(X, g, Wd, DIR == 0 ? 0 : 2, q, iL, jL, UL);
    recon_direct<K, Real>(X, g, Wd, DIR == 0 ? 1 : 3, q, iR, jR, UR);
  }
  Real pl, pr;
  if (DIR == 0) {
    riemann_x<Real>(g.riemann, UL, UR, gam, f, pl, pr);
  } else {
    Real a[4] = {UL[0], UL[2], UL[1], UL[3]};
    Real b[4] = {UR[0], UR[2], UR[1], UR[3]};
    Real h[4];
    riemann_x<Real>(g.riemann, a, b, gam, h, pl, pr);
    f[0] = h[0]; f[1] = h[2]; f[2] = h[1]; f[3] = h[3];
  }
  badL |= !(pos_finite(UL[0]) && pos_finite(pl));
  badR |= !(pos_finite(UR[0]) && pos_finite(pr));
  if (sUL) {
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      sUL[v] = UL[v];
      sUR[v] = UR[v];
    }
  }
}

// face between cell (iL,jL) and its neighbour (iR,jR) in direction DIR at radius K
template <int K, class Real, int DIR>
__device__ void face_at(const Real* X, const Grid& g, const DirectW<Real>& Wd, int iL, int jL,
                        Real* F, bool& badL, bool& badR) {
  constexpr int Q = rule_q(K);
  F[0] = F[1] = F[2] = F[3] = Real(0);
  badL = badR = false;
  // mirror pairs (g, -g) summed first, in the order of the first-pass sweep
#pragma unroll
  for (int kk = 0; kk < (Q + 1) / 2; ++kk) {
    Real f1[4];
    face_point<K, Real, DIR>(X, g, Wd, iL, jL, kk, f1, badL, badR);
    if (Q - 1 - kk != kk) {
      Real f2[4];
      face_point<K, Real, DIR>(X, g, Wd, iL, jL, Q - 1 - kk, f2, badL, badR);
#pragma unroll
      for (int v = 0; v < 4; ++v) F[v] = fma(Wd.w[K][kk], add_rn(f1[v], f2[v]), F[v]);
    } else {
#pragma unroll
      for (int v = 0; v < 4; ++v) F[v] = fma(Wd.w[K][kk], f1[v], F[v]);
    }
  }
}

// the flux and state-check bits of the face between (iL,jL) and its
// neighbour in direction DIR; a periodic seam face writes both copies
template <class Real, int DIR>
__device__ __forceinline__ void store_face(const StageArgs<Real>& A, const Grid& g, int iL,
                                           int jL, const Real* F, uint8_t bits) {
  const int iR = iL + (DIR == 0), jR = jL + (DIR == 1);
  if (DIR == 0) {
    int f = iR;  // face index
#pragma unroll
    for (int v = 0; v < 4; ++v) A.Fx[fxidx(g, v, f, jL)] = F[v];
    uint8_t* fb = A.fbx + (long long)jL * (g.nx + 1);
    fb[f] = (uint8_t)((fb[f] & kVerdictBits) | bits);
    if (g.periodic_x && (f == 0 || f == g.nx)) {
      int f2 = f == 0 ? g.nx : 0;
#pragma unroll
      for (int v = 0; v < 4; ++v) A.Fx[fxidx(g, v, f2, jL)] = F[v];
      fb[f2] = (uint8_t)((fb[f2] & kVerdictBits) | bits);
    }
  } else {
    int f = jR;
#pragma unroll
    for (int v = 0; v < 4; ++v) A.Fy[fyidx(g, v, iL, f)] = F[v];
    A.fby[(long long)f * g.nx + iL] = bits;
    if (g.periodic_y && (f == 0 || f == g.ny)) {
      int f2 = f == 0 ? g.ny : 0;
#pragma unroll
      for (int v = 0; v < 4; ++v) A.Fy[fyidx(g, v, iL, f2)] = F[v];
      A.fby[(long long)f2 * g.nx + iL] = bits;
    }
  }
}

// face f (0 W, 1 E, 2 S, 3 N) of queued cell c: recompute it if its EDP1
// radius changed; the face shared with another queued cell is done by the
// west/south one
// false when the face needs no work; else its left/lower cell (iL, jL) and
// its new EDP1 radius K
template <class Real>
__device__ __forceinline__ bool mood_face_plan(const StageArgs<Real>& A, const Grid& g,
                                               const Cascade& C, const uint32_t* stamp,
                                               uint32_t cur, int c, int f, int& iL, int& jL,
                                               int& K) {
  const int i = c % g.nx, j = c / g.nx;
  if (f >= 2 && g.dim == 1) return false;  // no y faces in 1D
  // every load of the decision depends on c alone: all are issued before
  // the first test, so that one memory latency covers them
  bool other = false;  // the face is the other queued cell's
  if (f == 0 || f == 2) {
    int nb = neighbour(g, i, j, f);
    other = nb >= 0 && stamp[nb] == cur;
  }
  iL = i;
  jL = j;
  if (f == 0) iL = i - 1;
  if (f == 2) jL = j - 1;
  const int iR = iL + (f < 2), jR = jL + (f >= 2);
  int nl, bl, nr, br;
  radius_pair(g, A.ord, stamp, cur, C, iL, jL, nl, bl);
  radius_pair(g, A.ord, stamp, cur, C, iR, jR, nr, br);
  if (other) return false;
  K = nl < nr ? nl : nr;
  const int Kold = bl < br ? bl : br;
  return K != Kold;  // else the EDP1 order of this face is unchanged
}

// what the MOOD kernel keeps in shared memory: the weights of the radii below
// the top (1 and 2 at most), which the lanes of a warp read at different
// radii, faces and points at once, in the slots of the radius-3 diamond (zero
// where a radius has no such point), and the states of each warp's points
template <class Real>
struct MoodShared {
  using Z = Real;
  Z z[2][4][3][kMaxN];
  Real st[8][32][8];  // [warp][point][left 0-3, right 4-7]
};
template <>
struct MoodShared<double> {
  using Z = int2;
  Z z[2][4][3][kMaxN];
  double st[8][32][8];
};
__device__ __forceinline__ void stage_mood_weights(const DirectW<double>& Wd, MoodShared<double>& S) {
  for (int k = threadIdx.x; k < 2 * 4 * 3 * kMaxN; k += blockDim.x) {
    const int m = k % kMaxN, q = k / kMaxN % 3, f = k / (3 * kMaxN) % 4, K = k / (12 * kMaxN);
    S.z[K][f][q][m] = Wd.z[K + 1][f][q][m];
  }
  __syncthreads();
}
__device__ __forceinline__ void stage_mood_weights(const DirectW<float>& Wd, MoodShared<float>& S) {
  for (int k = threadIdx.x; k < 2 * 4 * 3 * kMaxN; k += blockDim.x) {
    const int m = k % kMaxN, q = k / kMaxN % 3, f = k / (3 * kMaxN) % 4, K = k / (12 * kMaxN) + 1;
    // offset (a, b) of slot m: row starts 0, 1, 4, 9, 16, 21, 24
    const int b = m < 1 ? -3 : m < 4 ? -2 : m < 9 ? -1 : m < 16 ? 0 : m < 21 ? 1 : m < 24 ? 2 : 3;
    const int a = m - (b == -3 ? 0 : b == -2 ? 2 : b == -1 ? 6 : b == 0 ? 12 : b == 1 ? 18 : b == 2 ? 22 : 24);
    const int ab = (a < 0 ? -a : a) + (b < 0 ? -b : b);
    // the table's own order: rows b = -K..K
    int i = a + K - (b < 0 ? -b : b);
    for (int r = -K; r < b; ++r) i += 2 * (K - (r < 0 ? -r : r)) + 1;
    S.z[K - 1][f][q][m] = ab <= K ? Wd.z[K][f][q][i] : 0.0f;
  }
  __syncthreads();
}

// one variable of a face state at radius K <= 2 given at run time, from the
// weights in shared memory; all loads are issued before the first use.  FP32:
// recon_direct's sum, to which the points a radius lacks add zeros.
__device__ __forceinline__ double mood_value(const double* X, int pitch, const int2* z, int K,
                                             int off) {
  return fx_value<2>(X, pitch, z, K, off);
}
__device__ __forceinline__ float mood_value(const float* X, int pitch, const float* z, int K,
                                            int) {
  float x[stencil_n(2)];
  int k = 0;
#pragma unroll
  for (int b = -2; b <= 2; ++b)
#pragma unroll
    for (int a = -2; a <= 2; ++a) {
      const int ab = (a < 0 ? -a : a) + (b < 0 ? -b : b);
      if (ab <= 2) x[k++] = ab <= K ? X[(long long)b * pitch + a] : 0.0f;
    }
  float s = 0.0f;
  k = 0;
#pragma unroll
  for (int b = -2; b <= 2; ++b) {
    const int hb = 2 - (b < 0 ? -b : b), mid = k + hb;
    float t = mul_rn(z[diamond3_slot(0, b)], x[mid]);
#pragma unroll
    for (int a = 1; a <= 2; ++a)
      if (a <= hb)
        t = add_rn(t, add_rn(mul_rn(z[diamond3_slot(a, b)], x[mid + a]),
                             mul_rn(z[diamond3_slot(-a, b)], x[mid - a])));
    s = add_rn(s, t);
    k += 2 * hb + 1;
  }
  return s;
}

// entry k (0 itself, 1 W, 2 E, 3 S, 4 N) of queued cell c's neighbourhood:
// if c is the first queued cell of that cell's own list (itself, W, E, S,
// N), re-update it, re-detect it and return whether it is troubled; d gets
// the cell's index (or -1).  VL = 4: the four lanes of an aligned quad share
// an item, one variable each (6 FP64 instructions in a row for 24); the first
// detects and has the result.
template <int VL, class Real>
__device__ __forceinline__ bool mood_update_item(const StageArgs<Real>& A, const Grid& g,
                                                 const Detect& D, const Real* d2x,
                                                 const Real* d2y, StageC coef,
                                                 const uint32_t* stamp, uint32_t cur, int c,
                                                 int k, int& d) {
  const int v0 = VL == 4 ? threadIdx.x & 3 : 0;
  constexpr int NV = 4 / VL;
  const int i = c % g.nx, j = c / g.nx;
  d = k == 0 ? c : neighbour(g, i, j, k - 1);
  if (d < 0) return false;
  const int di = d % g.nx, dj = d / g.nx;
  // the loads of the ownership test and of the candidate depend on d alone:
  // all are issued before the test, so that one memory latency covers them
  bool taken = false;  // cell d is updated by another queued cell's item
  if (k > 0) {
    taken = stamp[d] == cur;
    // earlier entries of d's own list: W, E, S (in that order) before c
    const int back = k == 1 ? 1 : k == 2 ? 0 : k == 3 ? 3 : 2;
    for (int e = 0; e < 3; ++e) {
      if (e >= back) break;
      int o = neighbour(g, di, dj, e);
      taken |= o >= 0 && stamp[o] == cur;
    }
  }
  const long long wf = (long long)dj * (g.nx + 1) + di, sf = (long long)dj * g.nx + di;
  const unsigned bw = load_now(A.fbx + wf), be = load_now(A.fbx + wf + 1);
  const unsigned bs = load_now(A.fby + sf), bn = load_now(A.fby + sf + g.nx);
  const int od = (int)load_now(A.ord + d);
  const long long k0 = gidx(g, 0, di, dj);
  const bool with_u0 = __double_as_longlong(A.ca) != 0;
  double u0[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) u0[v] = with_u0 ? load_now(A.U0 + k0 + (v0 + v) * g.vstride) : 0.0;
  const Real r0 = load_now(A.Xr + k0), rw = load_now(A.Xr + k0 - 1), re = load_now(A.Xr + k0 + 1);
  const Real rs = load_now(A.Xr + k0 - g.pitch), rn = load_now(A.Xr + k0 + g.pitch);
  double y[NV];
  candidate<NV, Real>(A, g, di, dj, v0, coef, y);
  if (taken) {  // the same in all lanes of a quad
    d = -1;
    return false;
  }
  double Y[4];
  if constexpr (VL == 4) {
    const int lane = threadIdx.x & 31, base = lane & 28;
#pragma unroll
    for (int v = 0; v < 4; ++v) Y[v] = __shfl_sync(0xfu << base, y[0], base + v);
  } else {
#pragma unroll
    for (int v = 0; v < 4; ++v) Y[v] = y[v % NV];
  }
  bool flag = false;
  if (v0 == 0) {
    if (od != 0) {
      const int known = (int)(bw & kVerdictBits) >> 2;
      int verdict = known;
      // face_state_bad; the y faces' bits are zero in 1D
      flag = (((bw >> 1) | be | (bs >> 1) | bn) & 1) != 0;
      if (!flag) {
        auto lx = [&](int v, int a, int b) -> Real {
          if (v == 0 && a * a + b * b <= 1)
            return a < 0 ? rw : a > 0 ? re : b < 0 ? rs : b > 0 ? rn : r0;
          return xload<Real>(A.Xr, g, v, di + a, dj + b);
        };
        flag = troubled_at<Real>(lx, g, D, d2x, d2y, Y, verdict);
      }
      if (verdict != known) keep_verdict<Real>(A, g, di, dj, verdict);
    } else {
      Real f[4] = {(Real)Y[0], (Real)Y[1], (Real)Y[2], (Real)Y[3]};
      Real p = (Real)(g.gamma - 1.0) * (f[3] - Real(0.5) * (f[1] * f[1] + f[2] * f[2]) / f[0]);
      if (!(f[0] > Real(0)) || !(p > Real(0))) atomicAdd(&A.scw->nfog_pad[A.stage], 1);
    }
  }
  combine<NV, Real>(A, k0 + v0 * g.vstride, g.vstride, y, u0);
  return flag;
}

// ---------------------------------------------------------------------------
// the whole MOOD loop of one stage in one cooperative launch (Sec. 4 Step 10:
// repeat until no cell is flagged).  Every block takes part in every phase of
// every iteration, separated by grid-wide barriers:
//   lower the queued cells one cascade level  | barrier
//   recompute the faces whose EDP1 radius changed  | barrier
//   re-update + re-detect the queued cells and their face neighbours,
//   troubled ones into the other queue  | barrier
// and every block reads the new queue length to take the same decision.
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// barrier among `blocks` co-resident blocks on a running count of arrivals
// (never reset: the count at rest is a multiple of `blocks`): one atomic to
// arrive, and everyone polls for the count that completes the round.  A wait
// gives up as spin_limit.h says, after about a second without a change of
// *alive (null: none to look at), latches kErrSync and returns false; a block
// that sees the error leaves the loop, so no wait can outlast the limit.
__device__ __forceinline__ unsigned long long load_acquire(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ bool block_barrier(Scalars* sc, unsigned long long* count,
                                              unsigned blocks, const unsigned long long* alive,
                                              unsigned pause) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    volatile int* err = &sc->err;
    unsigned long long old;
    asm volatile("atom.add.acq_rel.gpu.global.u64 %0, [%1], 1;" : "=l"(old) : "l"(count) : "memory");
    const unsigned long long target = (old / blocks + 1) * blocks;
    int good = 1;
    spin_limit w;
    spin_start(&w, alive ? load_acquire(alive) : 0);
    while (load_acquire(count) < target) {
      const unsigned long long now = global_ns();
      if (spin_due(&w, now) &&
          ((*err & kErrSync) || spin_over(&w, now, alive ? load_acquire(alive) : 0))) {
        atomicOr(&sc->err, kErrSync);
        good = 0;
        break;
      }
      __nanosleep(pause);
    }
    if (*err & kErrSync) good = 0;
    ok = good;
  }
  __syncthreads();
  return ok != 0;
}
// of the whole grid
__device__ __forceinline__ bool grid_barrier(Scalars* sc) {
  return block_barrier(sc, &sc->bar_all, gridDim.x, nullptr, 20);
}

// Once a queue is short, the first kSmallBlocks blocks (on as many SMs) go on
// alone to the end of the loop, and once it is very short the first block:
// the others wait for them (or leave, without a tail).  A barrier among 32
// blocks takes 1.5-2 us, among all (about 300) 3-5; one block needs neither
// it nor the L1 invalidation that comes with it, and finds in L1 what the
// iteration before touched.  Chains of a few cells that walk along a
// discontinuity for hundreds of iterations are common.  They do not come
// back: a queue seldom grows, and stays correct if it does.
constexpr int kSmallBlocks = 32;
constexpr int kSmallQueue = 256;
constexpr int kOneQueue64 = 10, kOneQueue32 = 24;  // FP64, FP32

// the stamps of value v: two arrays, one per parity of v, so that an
// iteration can mark the cells of the next queue (value v + 1) while its own
// queue's marks (value v) are still being read
__device__ __forceinline__ uint32_t* stamp_of(const MoodArgs& M, uint32_t v) {
  return M.stamp + (long long)(v & 1u) * M.stamp_stride;
}

// problem of a pooled cell index gc: the handle's single problem
template <class Real>
struct SingleSite {
  const StageArgs<Real>& A;
  const Grid& g;
  const Detect& D;
  const Real* d2x;
  const Real* d2y;
  StageC* k;  // shared: the stage coefficients, three FP64 products for every item
  __device__ __forceinline__ void prepare() const {
    if (threadIdx.x == 0) *k = stage_coeffs<Real>(A, g, A.sc->dt);
  }
  __device__ __forceinline__ StageC coeffs(const StageArgs<Real>&, const Grid&) const { return *k; }
  template <class F>
  __device__ __forceinline__ void with(int gc, F&& f) const {
    f(A, g, D, d2x, d2y, 0);
  }
};

// a sign of life for the blocks that wait for the working ones: block 0, which
// always works, counts its trips through the phases' loops (fire and forget)
__device__ __forceinline__ void mood_progress(Scalars* sc, unsigned blocks) {
  if (blocks != gridDim.x && blockIdx.x == 0 && threadIdx.x == 0)
    asm volatile("red.relaxed.gpu.global.add.u64 [%0], 1;" ::"l"(&sc->progress) : "memory");
}

// lane index of a MOOD phase worked on by `blocks` blocks: the warps are
// ranked block-minor (warp 0 of every block, then warp 1, ...), so the few
// warps of a short iteration land on different SMs and FP64 sub-partitions
// instead of queueing on one
__device__ __forceinline__ long long mood_lane(unsigned blocks) {
  return ((long long)(threadIdx.x >> 5) * blocks + blockIdx.x) * 32 + (threadIdx.x & 31);
}

// the flux of a recomputed face from its points' fluxes, lane by lane: the
// four lanes of a face hold its points' fluxes fq and state checks bl, br;
// the first forms the Gauss sum in the order of face_at (mirror pairs summed
// first), so the flux is the same bit for bit.  Called by whole warps.
template <class Real>
__device__ __forceinline__ void gauss_sum(const DirectW<Real>& Wd, int K, const Real* fq, bool bl,
                                          bool br, Real* F, uint8_t& bits) {
  const int base = threadIdx.x & 28;
  Real fp[4][4];
#pragma unroll
  for (int p = 0; p < 4; ++p)
#pragma unroll
    for (int v = 0; v < 4; ++v) fp[p][v] = __shfl_sync(0xffffffffu, fq[v], base + p);
  const unsigned bbl = __ballot_sync(0xffffffffu, bl), bbr = __ballot_sync(0xffffffffu, br);
  // face_at's loop over (g, -g) pairs, one path for every rule size:
  // Q = 4: w1 (f1 + f2) + w0 (f0 + f3); Q = 3: w1 f1 + w0 (f0 + f2);
  // Q = 2: w0 (f0 + f1); Q = 1: w0 (f0 + 0), which rounds as w0 f0
  const int Q = rule_q(K);
  const Real w0 = Wd.w[K][0], w1 = Wd.w[K][1];
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    const Real z = Real(0);
    const Real last = Q == 4 ? fp[3][v] : Q == 3 ? fp[2][v] : Q == 2 ? fp[1][v] : z;
    const Real inner = fma(w0, add_rn(fp[0][v], last), z);
    const Real mid = Q == 4 ? add_rn(fp[1][v], fp[2][v]) : fp[1][v];
    const Real outer = fma(w1, mid, inner);
    F[v] = Q >= 3 ? outer : inner;
  }
  bits = (uint8_t)((((bbl >> base) & 0xFu) ? 1 : 0) | (((bbr >> base) & 0xFu) ? 2 : 0));
}

// The MOOD face recompute.  Point t of 16 n is point t % 4 of face (t / 4) % 4 of
// pooled cell queue[t / 16].  A warp takes P consecutive points (4, 8, 16 or
// 32, whole faces): lane l < P plans point l, then the eight values of a point
// (two sides, four variables) are reconstructed by eight lanes, four points at
// a time and every radius and direction alike, and lane l solves point l.  A
// point's chain is 8 times shorter than with one lane a point, and the 32
// lanes of an instruction cost what one does, so P is the number that makes
//   ceil(points / (P x sub-partitions)) x (a Riemann solve)
//   + P / 4 x (a reconstruction)
// smallest: short queues spread over the chip, long ones fill the lanes.
template <class Real, class Site>
__device__ __forceinline__ void mood_faces_phase(const Site& site, const MoodArgs& M,
                                                 const DirectW<Real>& Wd, MoodShared<Real>& S,
                                                 const Cascade& C, uint32_t cur,
                                                 const int* queue, int n, unsigned blocks) {
  constexpr bool F64 = sizeof(Real) == sizeof(double);
  const long long L = 16LL * n;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t* stamp = stamp_of(M, cur);
  // (in units of 100 cycles; the whole grid has two blocks an SM, the small
  // group one)
  const int subs = (blocks == gridDim.x && blocks > 1 ? 2 : 4) * blocks;
  int P = 4;
  long long best = 0;
#pragma unroll 1
  for (int p = 4; p <= 32; p *= 2) {
    const long long cost =
        (L + (long long)p * subs - 1) / ((long long)p * subs) * (F64 ? 28 : 5) + p / 4 * (F64 ? 6 : 3);
    if (p == 4 || cost < best) {
      best = cost;
      P = p;
    }
  }
  int off = 0;
  if constexpr (F64) off = Wd.off;
  const long long stride = (long long)blocks * (blockDim.x >> 5) * P;
  Real (*st)[8] = S.st[warp];
  for (long long t0 = ((long long)warp * blocks + blockIdx.x) * P; t0 < L; t0 += stride) {
    mood_progress(M.sc, blocks);
    const long long t = t0 + lane;
    const int q = (int)(t & 3);
    const int f = (int)((t >> 2) & 3);
    const bool mine = lane < P && t < L;
    const int gc = mine ? queue[t >> 4] : 0;
    int iL = 0, jL = 0, K = 0, pitch = 0;
    bool work = false;
    const Real* X = nullptr;  // the left cell, variable 0
    long long vs = 0;
    if (mine)
      site.with(gc, [&](const StageArgs<Real>& A, const Grid& g, const Detect&, const Real*,
                        const Real*, int first) {
        work = mood_face_plan<Real>(A, g, C, stamp + first, cur, gc - first, f, iL, jL, K);
        pitch = g.pitch;
        vs = g.vstride;
        X = A.Xr + gidx(g, 0, iL, jL);
      });
    const bool solve = work && q < rule_q(K);
    const int dir = f < 2 ? 0 : 1;
    const int plan = solve ? 1 | K << 1 | dir << 3 | q << 4 : 0;
#pragma unroll 1
    for (int p = 0; p < P; p += 4) {
      const int src = p + (lane >> 3), v = lane & 3, right = (lane >> 2) & 1;
      const int pl = __shfl_sync(0xffffffffu, plan, src);
      const Real* Xp = (const Real*)__shfl_sync(0xffffffffu, (unsigned long long)X, src);
      const long long vsp = __shfl_sync(0xffffffffu, vs, src);
      const int pp = __shfl_sync(0xffffffffu, pitch, src);
      if (pl) {
        const int k = (pl >> 1) & 3, d = (pl >> 3) & 1;
        Xp += v * vsp + (right ? (d ? pp : 1) : 0);
        st[src][lane & 7] =
            k == 0 ? *Xp : mood_value(Xp, pp, S.z[k - 1][2 * d + right][pl >> 4], k, off);
      }
    }
    __syncwarp();
    Real fq[4] = {Real(0), Real(0), Real(0), Real(0)};
    bool bl = false, br = false;
    if (solve) {
      // faces: 0 W, 1 E, 2 S, 3 N of the queued cell; the y direction swaps
      // the momenta around the x solver
      const int mn = 1 + dir, mt = 2 - dir;
      const Real* u = st[lane];
      const Real a[4] = {u[0], u[mn], u[mt], u[3]};
      const Real b[4] = {u[4], u[4 + mn], u[4 + mt], u[7]};
      Real h[4], pl, pr;
      site.with(gc, [&](const StageArgs<Real>& A, const Grid& g, const Detect&, const Real*,
                        const Real*, int) {
        riemann_x<Real>(g.riemann, a, b, (Real)g.gamma, h, pl, pr);
        // a recorded step keeps the states of the recomputed face
        if (A.sc->ctl.stape != nullptr) {
          const int qt = rule_q(Wd.top);
          if (dir == 0) tape_face<Real, 0>(A, g, qt, iL, jL, q, u, u + 4);
          else tape_face<Real, 1>(A, g, qt, iL, jL, q, u, u + 4);
        }
      });
      fq[0] = h[0];
      fq[1] = dir ? h[2] : h[1];
      fq[2] = dir ? h[1] : h[2];
      fq[3] = h[3];
      bl = !(pos_finite(a[0]) && pos_finite(pl));
      br = !(pos_finite(b[0]) && pos_finite(pr));
    }
    Real F[4];
    uint8_t bits;
    gauss_sum<Real>(Wd, K, fq, bl, br, F, bits);
    if (work && q == 0)
      site.with(gc, [&](const StageArgs<Real>& A, const Grid& g, const Detect&, const Real*,
                        const Real*, int) {
        if (dir == 0) store_face<Real, 0>(A, g, iL, jL, F, bits);
        else store_face<Real, 1>(A, g, iL, jL, F, bits);
      });
    __syncwarp();  // the states are read before the next points' are written
  }
}

// re-update + re-detect: item t is entry t % 5 (itself, W, E, S, N) of
// pooled cell queue[t / 5], VL lanes each; a cell found troubled is lowered
// one cascade level at once, marked with the next stamp and appended to the
// next queue
template <int VL, class Real, class Site>
__device__ __forceinline__ void mood_update_items(const Site& site, const MoodArgs& M,
                                                  const Cascade& C, uint32_t cur,
                                                  const int* queue, int n, int* next_queue,
                                                  int* next_count, unsigned blocks) {
  const long long stride = (long long)blocks * blockDim.x;
  const uint32_t* stamp = stamp_of(M, cur);
  uint32_t* next_stamp = stamp_of(M, cur + 1);
  for (long long l = mood_lane(blocks); l < 5LL * VL * n; l += stride) {
    mood_progress(M.sc, blocks);
    const int t = (int)(l / VL);
    const int gc = queue[t / 5];
    int dg = -1;
    bool flag = false;
    site.with(gc, [&](const StageArgs<Real>& A, const Grid& g, const Detect& D, const Real* d2x,
                      const Real* d2y, int off) {
      int d = -1;
      flag = mood_update_item<VL, Real>(A, g, D, d2x, d2y, site.coeffs(A, g), stamp + off, cur,
                                        gc - off, t % 5, d);
      if (flag) {
        // only this item updates cell d in this iteration: its radius and
        // its next stamp are written by no one else
        A.ord[d] = (uint8_t)C.next[A.ord[d]];
        next_stamp[off + d] = cur + 1;
      }
      dg = d >= 0 ? off + d : -1;
    });
    queue_push(flag, dg, next_queue, next_count);
  }
}
// four lanes an item where all find a thread at once, else one: the same FP64
// work, but detection on a quarter of the lanes
template <class Real, class Site>
__device__ __forceinline__ void mood_update_phase(const Site& site, const MoodArgs& M,
                                                  const Cascade& C, uint32_t cur,
                                                  const int* queue, int n, int* next_queue,
                                                  int* next_count, unsigned blocks) {
  if (20LL * n <= (long long)blocks * blockDim.x)
    mood_update_items<4, Real>(site, M, C, cur, queue, n, next_queue, next_count, blocks);
  else
    mood_update_items<1, Real>(site, M, C, cur, queue, n, next_queue, next_count, blocks);
}

// the loop itself, for one problem or a batch (Site); tail: every block has
// work to do after it, on the loop's results.  The first-pass queue
// is lowered and marked in a prologue; then every iteration is
//   recompute the faces whose EDP1 radius changed  | barrier
//   re-update + re-detect, lowering and marking the troubled cells
//   for the next iteration  | barrier
// and every block reads the new queue length to take the same decision.
template <class Real, class Site>
__device__ __forceinline__ void mood_loop_body(const Site& site, const MoodArgs& M,
                                               const DirectW<Real>& Wd, const Cascade& C,
                                               int stage, bool tail) {
  Scalars* sc = M.sc;
  const bool leader = blockIdx.x == 0 && threadIdx.x == 0;
  // the first pass filled queue 0; queue 1 receives the first iteration's
  // troubled cells (the counts are cleared here, used after a barrier).  Each
  // group of blocks has counts of its own, so a block that leaves the loop may
  // still read the old ones.
  __shared__ int one_next[2];
  int n = *(volatile int*)M.count;
  const int nfirst = n;
  int slot = 0, iters = 0, total = n;
  uint32_t cur = sc->stamp_cur + 1;  // stamp of the cells of the first queue
  const int cap = sc->ctl.max_iters;
  if (leader) sc->next[0][1] = sc->next[1][0] = sc->next[1][1] = 0;
  if (threadIdx.x == 0) one_next[0] = one_next[1] = 0;
  bool ok = true;
  unsigned blocks = gridDim.x;  // that work on the queue
  int* next = gridDim.x == 1 ? one_next : sc->next[0];
  auto barrier = [&]() {
    if (blocks == 1) {
      __syncthreads();
      return true;
    }
    return blocks == gridDim.x ? grid_barrier(sc)
                               : block_barrier(sc, &sc->bar_small, blocks, nullptr, 20);
  };
  // n decides who goes on; false: not this block
  constexpr int kOneQueue = sizeof(Real) == sizeof(double) ? kOneQueue64 : kOneQueue32;
  auto shrink = [&]() {
    if (blocks > 1 && n <= kOneQueue) {
      blocks = 1;
      next = one_next;
    } else if (blocks > (unsigned)kSmallBlocks && n <= kSmallQueue) {
      blocks = kSmallBlocks;
      next = sc->next[1];
    }
    return blockIdx.x < blocks;
  };
  __shared__ MoodShared<Real> MS;
  if (n > 0) {
    ok = shrink();
    if (ok) {
      site.prepare();  // for all threads after the barrier
      stage_mood_weights(Wd, MS);
      uint32_t* st = stamp_of(M, cur);
      for (long long q = mood_lane(blocks); q < n; q += (long long)blocks * blockDim.x) {
        const int gc = M.queue[0][q];
        site.with(gc, [&](const StageArgs<Real>& A, const Grid&, const Detect&, const Real*,
                          const Real*, int off) {
          A.ord[gc - off] = (uint8_t)C.next[A.ord[gc - off]];
        });
        st[gc] = cur;
      }
      ok = barrier();
    }
  }
  while (ok && n > 0) {
    if (iters >= cap) {
      if (leader) atomicOr(&sc->err, kErrCap);
      break;
    }
    if (!shrink()) break;
    const int* queue = M.queue[slot];
    mood_faces_phase(site, M, Wd, MS, C, cur, queue, n, blocks);
    if (!barrier()) break;
    mood_update_phase<Real>(site, M, C, cur, queue, n, M.queue[slot ^ 1], &next[slot ^ 1],
                            blocks);
    if (!barrier()) break;
    n = *(volatile int*)&next[slot ^ 1];
    // the queue just worked on receives the next iteration's cells
    if (leader) next[slot] = 0;
    total += n;
    iters += 1;
    slot ^= 1;
    cur += 1;
  }
  // the waiting blocks look at the leader's progress (mood_progress), so a long
  // loop is no timeout; the error flag of a failed wait also ends this one
  if (blocks != gridDim.x && tail)
    block_barrier(sc, &sc->bar_all, gridDim.x, &sc->progress, 256);
  if (leader) {
    sc->nbad_first[stage] = nfirst;
    sc->nbad_total[stage] = total;
    sc->iters[stage] = iters;
    sc->stamp_cur = cur;  // every value up to cur has been used
    // the queue is empty for the next stage, also after a failed loop
    *M.count = 0;
  }
}

// the loop's tail (LoopTail): every interior value of the stage output is
// final once the loop has ended (the last phase ended at a grid barrier, or
// the first pass, a previous kernel, wrote them all)
__device__ __forceinline__ void mood_loop_tail(const Grid& g, Scalars* sc, const LoopTail& T) {
  const long long tid = ((long long)(threadIdx.x >> 5) * gridDim.x + blockIdx.x) * 32 +
                        (threadIdx.x & 31);
  const long long stride = (long long)gridDim.x * blockDim.x;
  if (T.X) {
    const double t = sc->t + T.tfrac * sc->dt;
    const long long n = ghost_count(g);
    for (long long k = tid; k < n; k += stride) fill_ghost(T.X, T.Xf, g, t, k);
  }
  if (T.rate) {
    // as k_dt_reduce, for the next step: the maximum CFL rate over the cells
    double best = 0.0;
    bool bad = false;
    const long long n = (long long)g.nx * g.ny;
    for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += stride) {
      const int i = (int)(c % g.nx), j = (int)(c / g.nx);
      double a;
      if (!cell_rate_at(T.Xrate, T.Xfrate, g, i, j, a)) bad = true;
      else best = max_num(a, best);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0 && g.rate_floor > best) best = g.rate_floor;
    for (int o = 16; o > 0; o >>= 1) {
      const double ob = __shfl_xor_sync(0xffffffffu, best, o);
      best = max_num(ob, best);
    }
    bad = __any_sync(0xffffffffu, bad);
    if ((threadIdx.x & 31) == 0) {
      if (bad) atomicOr(&sc->rate_bad, 1);
      if (best > 0.0) atomicMax(&sc->rate_bits, (unsigned long long)__double_as_longlong(best));
    }
    // readers are later kernels: the flag can go up before every block is done
    if (blockIdx.x == 0 && threadIdx.x == 0) sc->rate_ready = 1;
  }
}

template <class Real>
__global__ void __launch_bounds__(256, 2) k_mood_loop(StageArgs<Real> A, MoodArgs M, Grid g,
                                                   Detect D,
                                                   const __grid_constant__ DirectW<Real> Wd,
                                                   Cascade C, int stage, LoopTail T) {
  pdl_wait();
  __shared__ StageC coef;
  const SingleSite<Real> site{A, g, D, Wd.d2x, Wd.d2y, &coef};
  mood_loop_body<Real>(site, M, Wd, C, stage, true);
  mood_loop_tail(g, M.sc, T);
}

// ---------------------------------------------------------------------------
// replay of a step with given radii (no detection): every face at the EDP1
// radius of a radius map, then candidate + RK combination
// ---------------------------------------------------------------------------
template <class Real, int DIR>
__global__ void __launch_bounds__(128) k_faces_frozen(StageArgs<Real> A, Grid g,
                                                      const __grid_constant__ DirectW<Real> Wd) {
  const long long nf = DIR == 0 ? (long long)(g.nx + 1) * g.ny : (long long)g.nx * (g.ny + 1);
  const long long f = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (f >= nf) return;
  int iL, jL;
  if (DIR == 0) {
    iL = (int)(f % (g.nx + 1)) - 1;
    jL = (int)(f / (g.nx + 1));
  } else {
    iL = (int)(f % g.nx);
    jL = (int)(f / g.nx) - 1;
  }
  const int iR = iL + (DIR == 0), jR = jL + (DIR == 1);
  auto rad = [&](int i, int j) -> int {
    if (i < 0 || i >= g.nx) {
      if (!g.periodic_x) return Wd.top;
      i = wrapi(i, g.nx);
    }
    if (j < 0 || j >= g.ny) {
      if (!g.periodic_y) return Wd.top;
      j = wrapi(j, g.ny);
    }
    return A.ord[cidx(g, i, j)];
  };
  const int a = rad(iL, jL), b = rad(iR, jR);
  const int K = a < b ? a : b;
  Real F[4];
  bool bl, br;
  switch (K) {
    case 0: face_at<0, Real, DIR>(A.Xr, g, Wd, iL, jL, F, bl, br); break;
    case 1: face_at<1, Real, DIR>(A.Xr, g, Wd, iL, jL, F, bl, br); break;
    case 2: face_at<2, Real, DIR>(A.Xr, g, Wd, iL, jL, F, bl, br); break;
    default: face_at<3, Real, DIR>(A.Xr, g, Wd, iL, jL, F, bl, br); break;
  }
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    if (DIR == 0) A.Fx[fxidx(g, v, iR, jL)] = F[v];
    else A.Fy[fyidx(g, v, iL, jR)] = F[v];
  }
}

template <class Real>
__global__ void __launch_bounds__(256) k_update_frozen(StageArgs<Real> A, Grid g) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  if (i >= g.nx || j >= g.ny) return;
  double Y[4];
  candidate<4, Real>(A, g, i, j, 0, stage_coeffs<Real>(A, g, A.sc->dt), Y);
  combine_store<Real>(A, g, i, j, Y);
}

// ---------------------------------------------------------------------------
// batched kernels: many independent problems of uneven sizes in one
// persistent launch per kernel class.  Each block walks a list of work items
// (problem, block coordinates); the problem's grid is staged in shared
// memory; all buffers are pooled, each problem at its own offsets.  A
// problem with dt = 0 (finished) only carries its state over.
// ---------------------------------------------------------------------------
template <class Real>
__device__ __forceinline__ StageArgs<Real> problem_args(const StageArgs<Real>& B, const Prob& P,
                                                        const Scalars* psc, int p) {
  StageArgs<Real> A = B;
  A.X = B.X + P.state_off;
  A.Xr = B.Xr + P.state_off;
  A.U0 = B.U0 + P.state_off;
  A.out = B.out + P.state_off;
  A.outr = B.outr ? B.outr + P.state_off : nullptr;
  A.W = B.W ? B.W + P.state_off : nullptr;
  A.out2 = B.out2 ? B.out2 + P.state_off : nullptr;
  A.Fx = B.Fx + P.fx_off;
  A.Fy = B.Fy + P.fy_off;
  A.fbx = B.fbx + P.fx_off / 4;  // face planes: one per variable in the flux pools
  A.fby = B.fby + P.fy_off / 4;
  A.ord = B.ord + P.cell_off;
  A.first = B.first + P.cell_off;
  A.sc = psc + p;
  return A;
}

template <class Real>
__device__ __forceinline__ const Real* d2_of(const Prob& P, int d);
template <>
__device__ __forceinline__ const double* d2_of<double>(const Prob& P, int d) {
  return d == 0 ? P.d2x : P.d2y;
}
template <>
__device__ __forceinline__ const float* d2_of<float>(const Prob& P, int d) {
  return d == 0 ? P.d2xf : P.d2yf;
}

// one block per work item: a software loop over items would let the
// compiler keep all parity weights in registers across items (they are loop
// invariant), doubling the register footprint; the block scheduler walks the
// item list instead
template <int R, class Real, int DIR, int FW>
__global__ void __launch_bounds__(32 * FW) k_faces_batch(StageArgs<Real> B, const Prob* probs,
                                                         const Scalars* psc, const Item* items,
                                                         const __grid_constant__ ParityW<Real> W) {
  pdl_wait();
  pdl_trigger();
  __shared__ FaceTile<R, Real, FW> tile;
  // the item's problem, read from shared memory on demand like kernel
  // parameters
  __shared__ Prob sp;
  __shared__ StageArgs<Real> sa;
  __shared__ int sw[3];
  if (threadIdx.x == 0 && threadIdx.y == 0) {
    const Item w = items[blockIdx.x];
    sp = probs[w.p];
    sa = problem_args<Real>(B, sp, psc, w.p);
    sw[0] = psc[w.p].dt == 0.0;  // finished problem
    sw[1] = w.a;
    sw[2] = w.b;
  }
  __syncthreads();
  if (sw[0]) return;  // uniform over the block
  faces_block<R, Real, DIR, FW>(sa, sp.g, W, sw[1], sw[2], tile);
}

// the fused x+y face kernel over (problem, segment, band) work items
template <int R, class Real>
__global__ void __launch_bounds__(32 * kXYRows, kXYBlocks) k_faces_xy_batch(
    StageArgs<Real> B, const Prob* probs, const Scalars* psc, const Item* items,
    const __grid_constant__ ParityW<Real> W) {
  pdl_wait();
  pdl_trigger();
  extern __shared__ __align__(16) unsigned char xy_smem[];
  XYShared<R, Real>& S = *reinterpret_cast<XYShared<R, Real>*>(xy_smem);
  __shared__ Prob sp;
  __shared__ StageArgs<Real> sa;
  __shared__ int sw[3];
  if (threadIdx.x == 0 && threadIdx.y == 0) {
    const Item w = items[blockIdx.x];
    sp = probs[w.p];
    sa = problem_args<Real>(B, sp, psc, w.p);
    sw[0] = psc[w.p].dt == 0.0;  // finished problem
    sw[1] = w.a;
    sw[2] = w.b;
  }
  __syncthreads();
  if (sw[0]) return;  // uniform over the block
  faces_xy_block<R, Real>(sa, sp.g, W, sw[1], sw[2], S);
}

template <class Real>
__global__ void __launch_bounds__(256) k_update_batch(StageArgs<Real> B, const Prob* probs,
                                                      const Scalars* psc, const Item* items,
                                                      int nitems,
                                                      const __grid_constant__ DirectW<Real> Wd) {
  __shared__ Prob sp;
  __shared__ StageArgs<Real> sa;
  __shared__ StageC sk;
  __shared__ int sw[3];
  const int tid = threadIdx.y * 32 + threadIdx.x;
  for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
    __syncthreads();
    if (tid == 0) {
      const Item w = items[it];
      sp = probs[w.p];
      sa = problem_args<Real>(B, sp, psc, w.p);
      sw[0] = psc[w.p].dt == 0.0;
      sw[1] = w.a;
      sw[2] = w.b;
      if (!sw[0]) sk = stage_coeffs<Real>(sa, sp.g, sa.sc->dt);
    }
    __syncthreads();
    const int i = sw[1] * 32 + threadIdx.x, j = sw[2] * 8 + threadIdx.y;
    if (sw[0]) {
      // finished: carry the state over unchanged
      if (i < sp.g.nx && j < sp.g.ny) {
#pragma unroll
        for (int v = 0; v < 4; ++v) sa.out[gidx(sp.g, v, i, j)] = sa.X[gidx(sp.g, v, i, j)];
      }
      continue;
    }
    update_cell_w<Real>(sa, sp.g, sp.det, Wd, d2_of<Real>(sp, 0), d2_of<Real>(sp, 1), i, j,
                        sp.cell_off, sk);
  }
}

// the first cells of a batch's problems in shared memory, where there is room:
// a search through the problems themselves is a chain of loads
constexpr int kMaxStarts = 512;
struct BatchStarts {
  int first[kMaxStarts];
};
// problem of a pooled cell index (probs sorted by cell_off)
__device__ __forceinline__ int problem_of(const Prob* probs, const BatchStarts& S, int nprob,
                                          int gc) {
  int lo = 0, hi = nprob - 1;
  while (lo < hi) {
    int mid = (lo + hi + 1) >> 1;
    if ((nprob <= kMaxStarts ? S.first[mid] : probs[mid].cell_off) <= gc) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// problem of a pooled cell index gc in a batch (problems sorted by their
// first cell)
template <class Real>
struct BatchSite {
  const StageArgs<Real>& B;
  const Prob* probs;
  const Scalars* psc;
  int nprob;
  const BatchStarts& starts;
  __device__ __forceinline__ void prepare() const {}
  __device__ __forceinline__ StageC coeffs(const StageArgs<Real>& A, const Grid& g) const {
    return stage_coeffs<Real>(A, g, A.sc->dt);
  }
  template <class F>
  __device__ __forceinline__ void with(int gc, F&& f) const {
    const int p = problem_of(probs, starts, nprob, gc);
    const Prob& P = probs[p];
    const StageArgs<Real> A = problem_args<Real>(B, P, psc, p);
    f(A, P.g, P.det, d2_of<Real>(P, 0), d2_of<Real>(P, 1), P.cell_off);
  }
};

template <class Real>
__global__ void __launch_bounds__(256, 2) k_mood_loop_batch(StageArgs<Real> B, MoodArgs M,
                                                         const Prob* probs, const Scalars* psc,
                                                         int nprob,
                                                         const __grid_constant__ DirectW<Real> Wd,
                                                         Cascade C, int stage) {
  __shared__ BatchStarts starts;
  for (int p = threadIdx.x; p < nprob && nprob <= kMaxStarts; p += blockDim.x)
    starts.first[p] = probs[p].cell_off;
  __syncthreads();
  const BatchSite<Real> site{B, probs, psc, nprob, starts};
  mood_loop_body<Real>(site, M, Wd, C, stage, false);
}

}  // namespace gpm
