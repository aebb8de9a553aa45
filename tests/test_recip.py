"""csrc/recip.h, the reciprocal of the Cholesky panels and the reflectors, on the host: the same header,
compiled with the host compiler (whose float division and fma are correctly rounded, as the device's
instructions are), against 1.0 / d."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2501_19090_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <random>
#include "recip.h"
static double worst = 0.0;
static long outside = 0, n = 0;
static void check(double d) {
  const double q = pifa::recip(d), ref = 1.0 / d;
  const int ex = (int)(pifa::bits_as<uint64_t>(d) >> 52);
  if (ex < 64 || ex > 1982) {  // the division itself
    outside += pifa::bits_as<uint64_t>(q) != pifa::bits_as<uint64_t>(ref);
    return;
  }
  // 1 / d - q = (1 - d q) / d, the numerator exact to a rounding; in units of 1 / d's last place
  const double err = std::fabs(std::fma(-d, q, 1.0)) / std::ldexp(d, 1022 - ex);
  const double ulp = std::ldexp(ref, ex - 1022) >= 2.0 ? std::ldexp(1.0, -51) : std::ldexp(1.0, -52);
  worst = std::fmax(worst, err / ulp);
  ++n;
}
int main() {
  std::mt19937_64 g(1);
  for (int i = 0; i < 2000000; ++i) check(pifa::bits_as<double>((uint64_t)(g() & 0x7fffffffffffffffull)));
  for (int ex = 0; ex < 2047; ++ex)  // around the powers of two, and both guard limits
    for (int64_t s = -64; s <= 64; ++s)
      if (ex > 0 || s > 0) check(pifa::bits_as<double>((uint64_t)(((int64_t)ex << 52) + s)));
  for (uint64_t t = 0; t < (1u << 23); ++t)  // every float32 significand, both ends of what is cut off
    for (int k = 0; k < 2; ++k) check(pifa::bits_as<double>((uint64_t)((1023ull << 52) | (t << 29) | (k ? 0x1fffffff : 0))));
  std::printf("%ld %.6f %ld\n", n, worst, outside);
}
"""


def test_reciprocal_is_within_0_501_units_of_the_division(tmp_path):
    src, exe = tmp_path / "recip_test.cpp", tmp_path / "recip_test"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    n, worst, outside = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    assert int(n) > 18_000_000 and float(worst) <= 0.501 and int(outside) == 0, (n, worst, outside)
