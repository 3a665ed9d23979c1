"""fxd_to_double of csrc/fixed_dot.h on the host at the ends of the range: a sum
beyond the largest double is not finite, one below it the double it should be,
small sums of large values and zeros come out as everywhere."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2110_08683_gb300", "csrc")

DRIVER = r"""
#include <float.h>
#include <math.h>
#include <stdio.h>
#include "fixed_dot.h"

static uint64_t st = 0x9e3779b97f4a7c15ull;
static double uni(void) {  /* splitmix64 */
  uint64_t z = (st += 0x9e3779b97f4a7c15ull);
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return (double)((z ^ (z >> 31)) >> 11) * 0x1p-53;
}
static double dot(int n, const double* z, const double* x, int T) {
  int E = FXD_EMIN;
  for (int i = 0; i < n; ++i) {
    const int e = (int)(fxd_hi(x[i]) >> 20) & 0x7ff;
    E = e > E ? e : E;
  }
  fxd_acc a = {0, 0, 0};
  for (int i = 0; i < n; ++i) {
    int32_t ch, cl;
    fxd_weight(z[i], T, &ch, &cl);
    const int64_t X = fxd_from_double(x[i], E);
    fxd_mac(&a, ch, cl, fxd_limb_hi(X), fxd_limb_lo(X));
  }
  return fxd_to_double(fxd_round(a), E, 63 - T, E == 0x7ff ? 0x7ff80000u : 0);
}

int main(void) {
  long bad = 0, n_checked = 0, over = 0;
  for (int t = 0; t < 200000; ++t) {
    /* three values, the largest at the top of the range or well below */
    const int top = t % 3 == 0 ? 1023 : 880 + t % 144;
    double z[3], x[3];
    _Float128 exact = 0;
    double m = 0;
    for (int i = 0; i < 3; ++i) {
      z[i] = (t & 1 ? 0.9 : 0.3) * (uni() - 0.2);
      x[i] = ldexp(1.0 + uni(), top - (int)(3 * uni()));
      if (t & 2) x[i] = -x[i];
      m = fmax(m, fabs(x[i]));
      exact += (_Float128)z[i] * x[i];
    }
    const double r = dot(3, z, x, 60), want = (double)exact;
    ++n_checked;
    int ok;
    if (isinf(want)) ok = !isfinite(r), ++over;
    else ok = fabs(want) > DBL_MAX * (1 - 0x1p-50) || fabs(r - want) <= m * 0x1p-57 + 0x1p-52 * fabs(want);
    if (!ok && bad++ < 5) printf("%a %a\n", r, want);
  }
  /* the largest double itself, and a constant of that size */
  const double one[2] = {0.5, 0.5}, big[2] = {DBL_MAX, DBL_MAX};
  bad += dot(2, one, big, 60) != DBL_MAX;
  /* zeros and cancelling sums of large values */
  const double pm[2] = {DBL_MAX, -DBL_MAX}, near[2] = {0x1p1000, -0x1.fffffffffffffp999};
  bad += dot(2, one, pm, 60) != 0.0;
  bad += dot(2, one, near, 60) != 0x1p946;
  /* weights beyond one (fewer bits): still the sum */
  const double w[2] = {300.0, -299.0}, c[2] = {0x1.8p1020, 0x1.8p1020}, c2[2] = {0x1.8p1020, -0x1.8p1020};
  bad += dot(2, w, c, 50) != 0x1.8p1020;
  bad += isfinite(dot(2, w, c2, 50));
  printf("checked %ld over %ld mismatches %ld\n", n_checked, over, bad);
  return bad != 0 || over == 0;
}
"""


def test_ends_of_the_range(tmp_path):
    src = tmp_path / "fxd.c"
    src.write_text(DRIVER)
    exe = tmp_path / "fxd"
    r = subprocess.run(["gcc", "-O2", "-std=gnu11", "-ffp-contract=off", "-I", CSRC, str(src),
                        "-o", str(exe), "-lm"], capture_output=True, text=True)
    if r.returncode:
        pytest.fail(r.stderr)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and "mismatches 0" in r.stdout, r.stdout
