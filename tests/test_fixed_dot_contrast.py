"""The fixed-point face states of csrc/fixed_dot.h with the method's own weights
where the outermost column of the stencil is up to 10^10 times the rest, so that
products of small weights decide: against binary128, and no less accurate (rms)
than the chain of FP64 FMAs that the sum stands for.

Bound, with m the stencil's largest |x|, n terms, L the sum of |z|: a value is
rounded to 2^-58 of a power of two <= m (half a unit), a weight to 2^-60, the sum
is cut to 2^-60 m, and rounded once to a double:
    |r - exact| <= m (L 2^-59 + n 2^-61 + 2^-60) + 2^-53 |r|."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2110_08683_gb300", "csrc")

DRIVER = r"""
#include <math.h>
#include <stdio.h>
#include "fixed_dot.h"
#include "gp_weights.h"

static uint64_t st = 0x9e3779b97f4a7c15ull;
static double uni(void) {  /* splitmix64 */
  uint64_t z = (st += 0x9e3779b97f4a7c15ull);
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return (double)((z ^ (z >> 31)) >> 11) * 0x1p-53;
}

static double dot(int n, const double* z, const double* x) {
  int E = FXD_EMIN;
  for (int i = 0; i < n; ++i) {
    const int e = (int)(fxd_hi(x[i]) >> 20) & 0x7ff;
    E = e > E ? e : E;
  }
  fxd_acc a = {0, 0, 0};
  for (int i = 0; i < n; ++i) {
    int32_t ch, cl;
    fxd_weight(z[i], 60, &ch, &cl);
    const int64_t X = fxd_from_double(x[i], E);
    fxd_mac(&a, ch, cl, fxd_limb_hi(X), fxd_limb_lo(X));
  }
  return fxd_to_double(fxd_round(a), E, 3, 0);
}

int main(void) {
  long bad = 0, n_checked = 0;
  for (int R = 1; R <= 3; ++R) {
    gpw_radius w;
    if (gpw_solve(R, 1.0, 1.0, 12.0, &w)) return 2;
    for (int lg = 0; lg <= 10; ++lg) {
      double s2 = 0, c2 = 0;
      for (int t = 0; t < 4000; ++t) {
        double x[25], m = 0;
        for (int i = 0; i < w.n; ++i) {
          x[i] = (1.0 + uni()) * (w.da[i] == -R ? pow(10, lg) : 1.0);
          m = fmax(m, x[i]);
        }
        for (int face = 0; face < 2; ++face)
          for (int k = 0; k < w.q; ++k) {
            const double* z = w.z[face][k];
            _Float128 exact = 0;
            double chain = 0, L = 0, size = 0;
            for (int i = 0; i < w.n; ++i) {
              exact += (_Float128)z[i] * x[i];
              chain = fma(z[i], x[i], chain);
              L += fabs(z[i]);
              size += fabs(z[i] * x[i]);
            }
            const double r = dot(w.n, z, x), e = (double)(r - exact), ec = (double)(chain - exact);
            const double lim = m * (L * 0x1p-59 + w.n * 0x1p-61 + 0x1p-60) + 0x1p-53 * fabs(r);
            ++n_checked;
            if (!(fabs(e) <= lim) && bad++ < 5) printf("R %d 1e%d err %g lim %g\n", R, lg, e, lim);
            s2 += e * e / (size * size);
            c2 += ec * ec / (size * size);
          }
      }
      if (!(s2 <= c2) && ++bad) printf("R %d 1e%d rms over the chain's %g\n", R, lg, sqrt(s2 / c2));
    }
  }
  printf("checked %ld mismatches %ld\n", n_checked, bad);
  return bad != 0;
}
"""


def test_contrast_against_binary128(tmp_path):
    src = tmp_path / "fxd.c"
    src.write_text(DRIVER)
    exe = tmp_path / "fxd"
    r = subprocess.run(["gcc", "-O2", "-std=gnu11", "-ffp-contract=off", "-I", CSRC, str(src),
                        os.path.join(CSRC, "gp_weights.c"), "-o", str(exe), "-lm"],
                       capture_output=True, text=True)
    if r.returncode:
        pytest.fail(r.stderr)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and "mismatches 0" in r.stdout, r.stdout
