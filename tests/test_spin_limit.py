"""When a wait between blocks gives up (csrc/spin_limit.h), on the host against
a simulated clock and progress word: never while the word moves at least once a
second, always within two seconds of its last move."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2110_08683_gb300", "csrc")

DRIVER = r"""
#include <stdio.h>
#include "spin_limit.h"

/* a wait polled every `step` ns from time `start` on; the word moves every
   `every` ns until `until` (ns after the start).  Returns the time after the
   start at which the wait gives up, or 0 if it has not by `end`. */
static uint64_t gives_up(uint64_t start, uint64_t step, uint64_t every, uint64_t until, uint64_t end) {
  spin_limit w;
  spin_start(&w, 7);
  for (uint64_t t = 0; t < end; t += step) {
    const uint64_t moved = t < until ? t : until;
    const uint64_t word = 7 + (every ? moved / every : 0);
    if (spin_due(&w, start + t) && spin_over(&w, start + t, word)) return t;
  }
  return 0;
}

int main(void) {
  const uint64_t s = 1000000000ull;
  int bad = 0;
  for (int k = 0; k < 2; ++k) {
    const uint64_t start = k ? 1ull << 60 : 0;
    /* nothing moves: a second */
    const uint64_t a = gives_up(start, 1000, 0, 0, 3 * s);
    bad += !(a >= s && a <= s + 2000);
    /* it moves more often than once a second: never */
    bad += gives_up(start, 10000, s * 9 / 10, 100 * s, 100 * s) != 0;
    bad += gives_up(start, 10000, s / 100, 100 * s, 100 * s) != 0;
    /* it moved for a while and stopped: between one and two seconds later */
    const uint64_t b = gives_up(start, 1000, s / 3, 5 * s, 20 * s);
    bad += !(b >= 5 * s && b <= 7 * s + 2000);
    const uint64_t c = gives_up(start, 1000, s / 3, s + s / 2, 20 * s);
    bad += !(c >= s + s / 2 && c <= 3 * s + s / 2 + 2000);
  }
  /* a clock that stands still: the polls end it */
  spin_limit w;
  spin_start(&w, 0);
  uint64_t n = 0;
  while (!(spin_due(&w, 5) && spin_over(&w, 5, 0))) ++n;
  bad += n != SPIN_LIMIT_POLLS;
  printf("mismatches %d\n", bad);
  return bad != 0;
}
"""


def test_gives_up_only_without_progress(tmp_path):
    src = tmp_path / "spin.c"
    src.write_text(DRIVER)
    exe = tmp_path / "spin"
    r = subprocess.run(["gcc", "-O2", "-std=gnu11", "-I", CSRC, str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    if r.returncode:
        pytest.fail(r.stderr)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and "mismatches 0" in r.stdout, r.stdout
