"""fxd_round of csrc/fixed_dot.h on the host: the rounded sum of the negated
terms is the negated sum, also where the sum lies within a hair of the middle
between two results (constructed: random terms meet that once in 2^28), and it
is within one unit of the exact sum, exact where the sum is a multiple of it."""
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

/* sum of C[i] s[i], the weights as fxd_weight makes them of C 2^-60 */
static int64_t rounded(int n, const int64_t* C, const int64_t* s, int sign) {
  fxd_acc a = {0, 0, 0};
  for (int i = 0; i < n; ++i) {
    int32_t ch, cl;
    fxd_weight(ldexp((double)C[i], -60), 60, &ch, &cl);
    fxd_mac(&a, ch, cl, fxd_limb_hi(sign * s[i]), fxd_limb_lo(sign * s[i]));
  }
  return fxd_round(a);
}

int main(void) {
  const int q = FXD_ROUND;
  const uint64_t low = (1ull << q) - 1;
  long bad = 0, n_checked = 0;
  for (int t = 0; t < 400000; ++t) {
    /* an odd C of at most 53 bits and its inverse modulo 2^q */
    int64_t C[3] = {(int64_t)((next() >> (11 + next() % 30)) | 1), 0, 0};
    uint64_t inv = (uint64_t)C[0];
    for (int k = 0; k < 6; ++k) inv *= 2 - (uint64_t)C[0] * inv;
    /* the wanted low bits of the sum: the middle, off it by little, or nothing */
    const uint64_t off = next() >> (20 + next() % 44);
    uint64_t want = t % 4 == 0 ? low / 2 + 1 : t % 4 == 1 ? low / 2 + 1 - off : t % 4 == 2 ? low / 2 + 1 + off : off;
    if (t % 32 == 3) want = 0;
    int64_t s[3] = {(int64_t)((want * inv) & low), 0, 0};
    if (t & 32) C[0] = -C[0];
    /* two more terms that change the limbs but not the sum's low bits */
    int n = 1;
    if (t & 64) {
      n = 3;
      C[1] = (1ll << 30) * (int64_t)(next() % (1 << 20) + 1);
      s[1] = (1ll << 30) * (int64_t)(next() % (1 << 20));
      if (next() & 1) s[1] = -s[1];
      C[2] = (int64_t)(next() >> 12);
      s[2] = (int64_t)1 << 58;
      if (next() & 1) s[2] = -s[2];
    }
    __int128 sum = 0;
    for (int i = 0; i < n; ++i) sum += (__int128)C[i] * s[i];
    const int64_t r = rounded(n, C, s, 1), m = rounded(n, C, s, -1);
    const __int128 err = ((__int128)r << q) - sum;
    const __int128 one = (__int128)1 << q;
    ++n_checked;
    if (r != -m || err >= one || err <= -one || ((sum & (one - 1)) == 0 && err != 0)) {
      if (bad++ < 5) printf("C %lld s %lld n %d: %lld and %lld\n", (long long)C[0], (long long)s[0], n, (long long)r, (long long)m);
    }
  }
  /* the same through the doubles */
  const double z = 0x1.4d723aa293814p-10, x = 0x1.9370488d23161p-1;
  double d[2];
  for (int k = 0; k < 2; ++k) {
    int32_t ch, cl;
    fxd_acc a = {0, 0, 0};
    fxd_weight(z, 60, &ch, &cl);
    const int E = 1022;
    const int64_t X = fxd_from_double(k ? -x : x, E);
    fxd_mac(&a, ch, cl, fxd_limb_hi(X), fxd_limb_lo(X));
    d[k] = fxd_to_double(fxd_round(a), E, 3, 0);
  }
  if (d[0] != -d[1] && ++bad) printf("%a %a\n", d[0], d[1]);
  printf("checked %ld mismatches %ld\n", n_checked, bad);
  return bad != 0;
}
"""


def test_round_is_odd(tmp_path):
    src = tmp_path / "fxd.c"
    src.write_text(DRIVER)
    exe = tmp_path / "fxd"
    r = subprocess.run(["gcc", "-O2", "-std=gnu11", "-ffp-contract=off", "-I", CSRC, str(src),
                        "-o", str(exe), "-lm"], capture_output=True, text=True)
    if r.returncode:
        pytest.fail(r.stderr)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and "mismatches 0" in r.stdout, r.stdout
