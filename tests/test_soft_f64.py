"""The integer-pipe division and square root (csrc/soft_f64.cuh) against the host's IEEE operations, bit for bit.

The header's routines are plain C++ apart from their seeds (single-precision 1/x and 1/sqrt(x)), which the host
form takes correctly rounded and then moves by a few units in the last place: the device's approximations are
within one unit.  Operands: random significands, significands near the ends of the range and near each other,
short ones, perfect squares, zeros, subnormals, infinities, NaN and the ends of the exponent range.
"""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = r"""
#define __host__
#define __device__
#define __forceinline__ inline
#include <cstdio>
#include "soft_f64.cuh"
using namespace hydro;
static uint64_t state;
static uint64_t rnd() {
  uint64_t z = (state += 0x9E3779B97F4A7C15ull);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}
static bool same(double a, double b) { return sf_bits(a) == sf_bits(b) || (a != a && b != b); }
int main() {
  const uint64_t MANT = 0xfffffffffffffull, SIGN = 1ull << 63;
  const double special[] = {0.0, -0.0, 1.0, -1.0, 5e-324, 2.2250738585072014e-308, 1.7976931348623157e308,
                            INFINITY, -INFINITY, NAN, 1e-310, 1.5};
  state = SEED;
  long bad = 0;
  for (double a : special)
    for (double b : special) bad += !same(soft_div(a, b), a / b) + !same(soft_sqrt(a), sqrt(a));
  for (long i = 0; i < 3000000; ++i) {
    uint64_t a = rnd(), b = rnd(), m = rnd(), fa = a & MANT, fb = b & MANT;
    switch (m & 7) {
      case 1: fa &= 0xff; break;
      case 2: fb |= 0xfffffffffff00ull; break;
      case 3: fa |= 0xffffffffff000ull; fb &= 0xfff; break;
      case 4: fb = (fa + ((m >> 8) & 15) - 8) & MANT; break;
      case 5: fa &= ~0xffffffull; fb &= ~0xfffffffull; break;
      case 6: fb = (m >> 8) & 3; fa = MANT - ((m >> 10) & 3); break;
      case 7: fa = (m >> 8) & 3; fb = MANT - ((m >> 10) & 3); break;
    }
    const uint64_t wide = (m >> 16) & 1, span = wide ? 2048 : 200, lo = wide ? 0 : 923;
    const double x = sf_double((a & SIGN) | ((lo + (m >> 20) % span) << 52) | fa);
    const double y = sf_double((b & SIGN) | ((lo + (m >> 40) % span) << 52) | fb);
    bad += !same(soft_div(x, y), x / y) + !same(soft_sqrt(fabs(x)), sqrt(fabs(x))) + !same(soft_sqrt(x), sqrt(x));
    const double z = (double)((uint64_t)(a >> 37)) * (double)((uint64_t)(a >> 37));
    bad += !same(soft_sqrt(z), sqrt(z));
  }
  printf("%ld\n", bad);
  return bad != 0;
}
"""


@pytest.mark.parametrize("ulp", [-2, -1, 0, 1, 2])
def test_division_and_square_root_round_as_ieee(tmp_path, ulp):
    src = tmp_path / "check.cpp"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "check")
    subprocess.run(["g++", "-O2", "-ffp-contract=off", "-std=c++17", f"-DSOFT_SEED_ULP={ulp}", f"-DSEED={ulp + 11}",
                    "-I", os.path.join(ROOT, "paper_1306_6883_gb300", "csrc"), "-o", exe, str(src)], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
