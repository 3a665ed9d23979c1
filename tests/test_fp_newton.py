"""The integer-pipe reciprocal and square root of csrc/fp_newton.h on the
host, with seeds as far off as the hardware's approximations may be (2^-22
relative, twice the documented errors), against extended precision.

Bound: half a unit in the last place from the rounding, plus what the
fixed-point steps leave: the reciprocal's last residual is cut at 2^-59
(2^25 of 2^84) of at most one and its correction at 2^-62 of [1/2, 1), the
square of the first step's error (seed error^2 + 2 roundings, below 2^-30)
adds 2^-60: together below 2^-57, 0.04 units.  The square root's residual
and correction are cut at 2^-59 and 2^-62 of [1, 2), its step's error adds
2^-61: below 2^-58, 0.02 units."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2110_08683_gb300", "csrc")

DRIVER = r"""
#include <math.h>
#include <stdio.h>
#include "fp_newton.h"

static uint64_t st = 0x9e3779b97f4a7c15ull;
static uint64_t next(void) {  /* splitmix64 */
  uint64_t z = (st += 0x9e3779b97f4a7c15ull);
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}
static double uni(void) { return (double)(next() >> 11) * 0x1p-53; }
static double ulps(long double got, long double want) {
  return (double)(fabsl(got - want) / ldexpl(1.0L, ilogbl(want) - 52));
}

int main(void) {
  double wr = 0, ws = 0;
  for (long t = 0; t < 4000000; ++t) {
    /* random significands, and those next to powers of two and to zero tails */
    uint64_t m = next() & 0xfffffffffffffull;
    switch (t % 6) {
      case 0: m = 0; break;
      case 1: m = 0xfffffffffffffull - (next() & 15); break;
      case 2: m = next() & 15; break;
      case 3: m &= 0xfffff00000000ull; break;
      default: break;
    }
    /* every normal exponent whose reciprocal is normal */
    const uint64_t e = t % 5 ? 1003 + next() % 41 : 2 + next() % 2042, b = m | e << 52;
    double x;
    memcpy(&x, &b, 8);
    const int end = t % 7 < 2; /* the seed's error at its end, or anywhere */
    const double off = end ? (t % 7 ? 0x1p-22 : -0x1p-22) : (2 * uni() - 1) * 0x1p-22;
    const float rs = (float)(1.0 / (double)fpn_recip_arg(x) * (1 + off));
    const double r = t & 1 ? fpn_recip_seeded(x, rs) : -fpn_recip_seeded(-x, rs);
    wr = fmax(wr, ulps(r, 1.0L / x));
    const float qs = (float)(1.0 / sqrt((double)fpn_sqrt_arg(x)) * (1 + off));
    ws = fmax(ws, ulps(fpn_sqrt_seeded(x, qs), sqrtl(x)));
  }
  printf("recip %.4f sqrt %.4f\n", wr, ws);
  return !(wr <= 0.54 && ws <= 0.52);
}
"""


def test_reciprocal_and_square_root_within_their_bounds(tmp_path):
    src = tmp_path / "fpn.c"
    src.write_text(DRIVER)
    exe = tmp_path / "fpn"
    r = subprocess.run(["gcc", "-O2", "-std=gnu11", "-ffp-contract=off", "-I", CSRC, str(src),
                        "-o", str(exe), "-lm"], capture_output=True, text=True)
    if r.returncode:
        pytest.fail(r.stderr)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
