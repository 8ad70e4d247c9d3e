"""The integer-pipe FP64 operations (csrc/soft_f64.cuh: division, square root, comparisons, minima, scalings by
two) against the host's IEEE operations, bit for bit.

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
#include <cmath>
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
// the smaller, or the number where the other is a NaN of either kind (CUDA's fmin; the host's takes a signalling
// NaN as the result)
static double min_num(double a, double b) { return a != a ? b : b != b || a < b ? a : b; }
static long helpers(double a, double b) {
  const double p = fabs(a), q = fabs(b), c = 1e-10;
  long bad = 0;
  bad += sf_zero(a) != (a == 0) || sf_gt0(a) != (a > 0) || sf_lt0(a) != (a < 0) || sf_ge0(a) != (a >= 0) ||
         sf_le0(a) != (a <= 0) || sf_finite(a) != std::isfinite(a);
  bad += !same(sf_abs(a), fabs(a)) + !same(sf_neg(a), -a) + !same(sf_min_nonneg(p, q), min_num(p, q));
  bad += (sf_le_nonneg(p, q) != (p <= q)) + (sf_lt_nonneg(p, q) != (p < q));
  bad += !same(sf_floor_at(a, c), a < c ? c : a) + !same(sf_half(a), 0.5 * a) + !same(sf_twice(a), 2.0 * a);
  return bad + (sf_same_sign(a, b) != (a * b > 0));
}
int main() {
  const uint64_t MANT = 0xfffffffffffffull, SIGN = 1ull << 63;
  const double special[] = {0.0, -0.0, 1.0, -1.0, 5e-324, 2.2250738585072014e-308, 1.7976931348623157e308,
                            INFINITY, -INFINITY, NAN, 1e-310, 1.5};
  state = SEED;
  long bad = 0;
  for (double a : special)
    for (double b : special) bad += !same(soft_div(a, b), a / b) + !same(soft_sqrt(a), sqrt(a)) + helpers(a, b);
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
    bad += helpers(x, y);
    const double z = (double)((uint64_t)(a >> 37)) * (double)((uint64_t)(a >> 37));
    bad += !same(soft_sqrt(z), sqrt(z));
  }
  printf("%ld\n", bad);
  return bad != 0;
}
"""


@pytest.mark.parametrize("ulp", [-2, -1, 0, 1, 2])
def test_integer_pipe_operations_equal_ieee(tmp_path, ulp):
    src = tmp_path / "check.cpp"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "check")
    subprocess.run(["g++", "-O2", "-ffp-contract=off", "-std=c++17", f"-DSOFT_SEED_ULP={ulp}", f"-DSEED={ulp + 11}",
                    "-I", os.path.join(ROOT, "paper_1306_6883_gb300", "csrc"), "-o", exe, str(src)], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
