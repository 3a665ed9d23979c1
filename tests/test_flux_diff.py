"""The float operations of csrc/fp_bits.h that stand for FP64 ones, on the
host: the double difference of two floats and the product with a power of two,
where each says that it holds.  Each must give the bits of the FP64 operation."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2110_08683_gb300", "csrc")

DRIVER = r"""
#include <math.h>
#include <stdio.h>
#include "fp_bits.h"

static uint64_t st = 0x243f6a8885a308d3ull;
static uint64_t next(void) {  /* splitmix64 */
  uint64_t z = (st += 0x9e3779b97f4a7c15ull);
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}
static long bad = 0, n = 0, exact = 0, other = 0;
static void same(double want, double got, const char* what) {
  ++n;
  if (isnan(want) ? !isnan(got) : fpb_bits_of_double(want) != fpb_bits_of_double(got)) {
    if (bad++ < 10) printf("%s: want %a got %a\n", what, want, got);
  }
}
static void diff(float a, float b) {
  int ok;
  const double got = fpb_diff(a, b, &ok);
  if (ok) {
    ++exact;
    same((double)a - (double)b, got, "difference");
  } else {
    ++other;
  }
}
static void times(double x, double c, const char* what) {
  if (fpb_pow2_steps(x, c)) same(x * c, fpb_step_exponent(x, c), what);
  else ++other;
}
static float flt(void) { return fpb_float_of_bits((uint32_t)next()); }
int main(void) {
  for (int k = 0; k < 2000000; ++k) {
    const float a = flt();
    diff(a, flt());
    /* neighbours in size, among them the exact ones */
    uint32_t b;
    memcpy(&b, &a, 4);
    diff(a, fpb_float_of_bits(b + (uint32_t)(next() >> (33 + next() % 31))));
    /* exponents up to 40 apart, either sign: the error term in every position */
    diff(a, ldexpf(1.0f + (float)(next() >> 41) * 0x1p-23f, (int)(next() % 81) - 40) *
                (next() & 1 ? a : -a));
    diff(ldexpf(1.0f, (int)(next() % 200) - 100), ldexpf((float)(next() >> 40), (int)(next() % 200) - 130));
    diff(a, fpb_float_of_bits((b ^ 0x80000000u) + (uint32_t)(next() % 5)));
    /* a power of two times any double, and one at the ends of the range */
    const double c = ldexp(1.0, (int)(next() % 2046) - 1022);
    const double x = fpb_double_of_bits(next());
    const double ends[] = {ldexp(1.0 + (double)(next() % 1024) / 1024.0, -1022 + (int)(next() % 4)),
                           0x1.fffffffffffffp1023, fpb_double_of_bits(next() >> 12)};
    if (!fpb_is_pow2(c) || fpb_is_pow2(c * 1.5) || fpb_is_pow2(-c)) ++bad;
    times(x, c, "product");
    for (int e = 0; e < 3; ++e) times(ends[e], 0.25, "quarter");
  }
  const float sp[] = {0.0f, -0.0f, INFINITY, -INFINITY, NAN, 1.0f, -1.0f, 0x1p-149f, 0x1p-126f,
                      0x1.fffffep127f, -0x1.fffffep127f, 0x1p-24f};
  for (int i = 0; i < 12; ++i)
    for (int j = 0; j < 12; ++j) {
      diff(sp[i], sp[j]);
      times((double)sp[i], 0.5, "half");
    }
  if (exact < n / 4 || other > n) ++bad;
  printf("%ld checked, %ld exact differences, %ld bad\n", n, exact, bad);
  return bad != 0;
}
"""


def test_float_operations(tmp_path):
    src = tmp_path / "t.c"
    src.write_text(DRIVER)
    exe = tmp_path / "t"
    subprocess.run(["gcc", "-O2", "-I", CSRC, str(src), "-o", str(exe), "-lm"], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout
