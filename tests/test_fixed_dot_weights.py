"""fxd_weight of csrc/fixed_dot.h on the host: a weight becomes the nearest
multiple of 2^-T, exactly itself where it is one."""
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

int main(void) {
  long bad = 0, n_checked = 0;
  for (int t = 0; t < 400000; ++t) {
    const int T = 57 + t % 4;
    double c = ldexp((double)((next() >> 11) | 0x10000000000000ull), -53 - (int)(next() % 40));
    if (c >= 1.0 - 0x1p-30) c *= 0.5;
    if (t & 4) c = -c;
    int32_t hi, lo;
    fxd_weight(c, T, &hi, &lo);
    const __int128 C = ((__int128)hi << FXD_SPLIT) + lo;
    const _Float128 off = (_Float128)C - (_Float128)c * (_Float128)ldexp(1.0, T);
    ++n_checked;
    if (off > 0.5 || off < -0.5 || lo > 1 << (FXD_SPLIT - 1) || lo < -(1 << (FXD_SPLIT - 1))) {
      if (bad++ < 5) printf("T %d c %a off %g\n", T, c, (double)off);
    }
  }
  printf("checked %ld mismatches %ld\n", n_checked, bad);
  return bad != 0;
}
"""


def test_weights_are_the_nearest(tmp_path):
    src = tmp_path / "fxd.c"
    src.write_text(DRIVER)
    exe = tmp_path / "fxd"
    r = subprocess.run(["gcc", "-O2", "-std=gnu11", "-ffp-contract=off", "-I", CSRC, str(src),
                        "-o", str(exe), "-lm"], capture_output=True, text=True)
    if r.returncode:
        pytest.fail(r.stderr)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and "mismatches 0" in r.stdout, r.stdout
