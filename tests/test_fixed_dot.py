"""The fixed-point stencil sums of csrc/fixed_dot.h on the host, against
binary128 sums of the same doubles.

Bound, with m the stencil's largest |x|, n terms, L the sum of |z|: a value
is cut off below 2^-56 m (nothing is cut where every value is within a
factor of 16 of m or zero), a weight is rounded to 2^-60 (half a unit each),
the sum to 2^-60 m, and once to a double:
    |r - exact| <= m (L 2^-56 [cut] + n 2^-61 + 2^-60) + 2^-53 |r|."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2110_08683_gb300", "csrc")

DRIVER = r"""
#include <math.h>
#include <stdio.h>
#include "fixed_dot.h"

static uint64_t st = 0x9e3779b97f4a7c15ull;
static uint64_t next(void) {  /* splitmix64 */
  uint64_t z = (st += 0x9e3779b97f4a7c15ull);
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}
static double uni(void) { return (double)(next() >> 11) * 0x1p-53; }

static double dot(int n, const double* z, const double* x, int T, int reverse, int negate) {
  int E = FXD_EMIN;
  for (int i = 0; i < n; ++i) {
    const int e = (int)(fxd_hi(x[i]) >> 20) & 0x7ff;
    E = e > E ? e : E;
  }
  fxd_acc a = {0, 0, 0};
  for (int k = 0; k < n; ++k) {
    const int i = reverse ? n - 1 - k : k;
    int32_t ch, cl;
    fxd_weight(z[i], T, &ch, &cl);
    const int64_t X = fxd_from_double(negate ? -x[i] : x[i], E);
    fxd_mac(&a, ch, cl, fxd_limb_hi(X), fxd_limb_lo(X));
  }
  return fxd_to_double(fxd_round(a), E, 63 - T, E == 0x7ff ? 0x7ff80000u : 0);
}

int main(void) {
  long bad = 0, n_checked = 0;
  for (int t = 0; t < 200000; ++t) {
    const int n = t % 4 == 0 ? 5 : t % 4 == 1 ? 13 : 25;
    double z[25], x[25], sum = 0, L = 0, m = 0, small = HUGE_VAL;
    for (int i = 0; i < n; ++i) sum += z[i] = uni() - 0.3;
    for (int i = 0; i < n; ++i) z[i] /= fabs(sum) < 1 ? 1 : sum;
    /* contrast 1 to 2^60 between neighbours, either sign, some zeros, any scale */
    const int range = (int)(next() % 5) * 15;
    const double scale = ldexp(1.0, (int)(next() % 1600) - 800);
    for (int i = 0; i < n; ++i) {
      x[i] = scale * ldexp(1.0 + uni(), -(int)(next() % (range + 1)));
      if (t & 8) x[i] = next() & 1 ? -x[i] : x[i];
      if ((t & 48) == 48 && next() % 4 == 0) x[i] = 0;
    }
    double big = 0;
    for (int i = 0; i < n; ++i) {
      L += fabs(z[i]);
      big = fmax(big, fabs(z[i]));
      m = fmax(m, fabs(x[i]));
      if (x[i] != 0) small = fmin(small, fabs(x[i]));
    }
    int T = 60;
    while (ldexp(big, T - 60) >= 1 - 0x1p-30 || ldexp(L, T - 60) >= 3.9) --T;
    _Float128 exact = 0;
    for (int i = 0; i < n; ++i) exact += (_Float128)z[i] * x[i];
    const double r = dot(n, z, x, T, 0, 0);
    const double cut = m <= 8 * small ? 0 : L * 0x1p-56;
    const double lim = m * (cut + ldexp(n, -1 - T) + ldexp(1, -T)) + 0x1p-53 * fabs(r);
    const double err = (double)(r > exact ? r - exact : exact - r);
    ++n_checked;
    if (!(err <= lim)) {
      if (bad++ < 5) printf("n %d err %g lim %g\n", n, err, lim);
    }
    /* no order, and odd */
    if (dot(n, z, x, T, 1, 0) != r || dot(n, z, x, T, 0, 1) != -r) {
      if (bad++ < 5) printf("order or sign\n");
    }
  }
  /* weights that sum to one give a constant back exactly */
  for (int t = 0; t < 20000; ++t) {
    const double c = ldexp(1.0 + uni(), (int)(next() % 100) - 50) * (next() & 1 ? 1 : -1);
    const double z[5] = {0.625, -0.375, 0.5, 0.375, -0.125}, x[5] = {c, c, c, c, c};
    if (dot(5, z, x, 60, 0, 0) != c && bad++ < 5) printf("constant %a\n", c);
  }
  /* zeros (of either sign) give zero; a NaN or an infinity gives a NaN */
  const double z2[2] = {0.5, 0.5}, zz[2] = {0.0, -0.0}, inf[2] = {1.0, HUGE_VAL}, nan2[2] = {NAN, 2.0};
  if (dot(2, z2, zz, 60, 0, 0) != 0.0) ++bad;
  if (!isnan(dot(2, z2, inf, 60, 0, 0)) || !isnan(dot(2, z2, nan2, 60, 0, 0))) ++bad;
  printf("checked %ld mismatches %ld\n", n_checked, bad);
  return bad != 0;
}
"""


def test_fixed_point_sums_against_binary128(tmp_path):
    src = tmp_path / "fxd.c"
    src.write_text(DRIVER)
    exe = tmp_path / "fxd"
    r = subprocess.run(["gcc", "-O2", "-std=gnu11", "-ffp-contract=off", "-I", CSRC, str(src),
                        "-o", str(exe), "-lm"], capture_output=True, text=True)
    if r.returncode:
        pytest.fail(r.stderr)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and "mismatches 0" in r.stdout, r.stdout
