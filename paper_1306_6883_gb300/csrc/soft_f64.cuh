// IEEE double division and square root on the integer pipes, correctly rounded: the same bits as a / b and
// sqrt(x) for every input.
//
// Why: a GB300 SM executes a warp's FP64 instruction in 16 cycles on one unit shared by its four sub-cores,
// against 2 cycles on each sub-core for an integer one, and a division or square root is a chain of about nine
// FP64 instructions.  Measured per SM sub-core (cycles per warp operation, 304 blocks of 512 threads): FP64 add,
// multiply 65-77, division 556, square root 580, 32-bit integer add, logic, shift 2.2, multiply 2.2, multiply
// high 4.2.  The routines below are about 45 integer instructions.  The FP64 step spent more than half of its
// FP64 instructions in them: KH 512^2 30.9 M -> 13.7 M FP64 warp instructions per launch, 2.15 -> 1.15 ms (ncu);
// KH 1024^2 6.52 -> 3.38 ms per step.
//
// Method: a significand quotient (root) of 54 bits from a 32-bit reciprocal (reciprocal root) v: the hardware's
// single-precision approximation, one Newton step in 32-bit fixed point, then 31 bits and 23 more bits of the
// result, each from v and an exact remainder (64-bit wrap-around arithmetic: the remainders themselves are
// small).  With a seed within 2^-21 of the reciprocal, v is within 5 units of 2^-32 of it, the first partial
// result within 12 units of 2^-30, and the sum of both within 0.9 of a unit of the 54-bit result q.  Rounding
// then needs no more than the sign of the last remainder: the result rounded to 53 bits is (q + (r >= 0)) / 2,
// since an even q is not near a rounding boundary and neither operation has exact ties (Markstein's "IA-64 and
// Elementary Functions" gives the argument for both).
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

namespace hydro {

// Host forms of the device primitives let a plain C++ program check the routines (__host__ and the like then
// defined away); SOFT_SEED_ULP moves the seeds by that many units in the last place.
#ifndef SOFT_SEED_ULP
#define SOFT_SEED_ULP 0
#endif

#define HYDRO_HD __host__ __device__ __forceinline__

HYDRO_HD uint32_t sf_umulhi(uint32_t a, uint32_t b) {
#ifdef __CUDA_ARCH__
  return __umulhi(a, b);
#else
  return (uint32_t)(((uint64_t)a * b) >> 32);
#endif
}
// high word of a (signed) * b (unsigned)
HYDRO_HD int32_t sf_mulhi_su(int32_t a, uint32_t b) {
#ifdef __CUDA_ARCH__
  int32_t r;  // b - 2^32 as a signed operand for b >= 2^31, which the added a makes up for
  asm("mad.hi.s32 %0, %1, %2, %1;" : "=r"(r) : "r"(a), "r"((int32_t)b));
  return r;
#else
  return (int32_t)(((int64_t)a * (int64_t)b) >> 32);
#endif
}
// single-precision 1/x and 1/sqrt(x) of the float with these bits, as bits
HYDRO_HD uint32_t sf_rcp_seed(uint32_t bits) {
#ifdef __CUDA_ARCH__
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(__uint_as_float(bits)));
  return __float_as_uint(r);
#else
  float f, r;
  memcpy(&f, &bits, 4);
  r = (float)(1.0 / f);
  memcpy(&bits, &r, 4);
  return bits + SOFT_SEED_ULP;
#endif
}
HYDRO_HD uint32_t sf_rsqrt_seed(uint32_t bits) {
#ifdef __CUDA_ARCH__
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(__uint_as_float(bits)));
  return __float_as_uint(r);
#else
  float f, r;
  memcpy(&f, &bits, 4);
  r = (float)(1.0 / sqrt((double)f));
  memcpy(&bits, &r, 4);
  return bits + SOFT_SEED_ULP;
#endif
}
HYDRO_HD uint64_t sf_bits(double x) {
#ifdef __CUDA_ARCH__
  return (uint64_t)__double_as_longlong(x);
#else
  uint64_t u;
  memcpy(&u, &x, 8);
  return u;
#endif
}
HYDRO_HD double sf_double(uint64_t u) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)u);
#else
  double x;
  memcpy(&x, &u, 8);
  return x;
#endif
}
HYDRO_HD uint32_t sf_hi(uint64_t u) { return (uint32_t)(u >> 32); }
HYDRO_HD uint32_t sf_lo(uint64_t u) { return (uint32_t)u; }

// Quotient of two normal numbers (exponent fields ea, eb) whose quotient is a normal number.
HYDRO_HD double soft_div_core(uint64_t ua, uint64_t ub, int32_t ea, int32_t eb) {
  const uint64_t mb = (ub & 0xfffffffffffffull) | 0x10000000000000ull;
  uint64_t ma = (ua & 0xfffffffffffffull) | 0x10000000000000ull;
  const bool less = ma < mb;  // scale the numerator so that ma / mb is in [1, 2)
  ma = less ? ma << 1 : ma;
  const int32_t e = ea - eb + 1022 - (less ? 1 : 0);
  const uint32_t Bh = (uint32_t)(mb >> 21);
  uint32_t y = sf_rcp_seed(0x3f800000u | ((uint32_t)(mb >> 29) & 0x7fffffu));
  y = y > 0x3f7fffffu ? 0x3f7fffffu : y;
  y = y < 0x3f000000u ? 0x3f000000u : y;
  const uint32_t v0 = (y << 8) | 0x80000000u;  // 2^32 / (mb / 2^52)
  const int32_t err = (int32_t)(0x80000000u - sf_umulhi(Bh, v0));
  const uint32_t v = v0 + (uint32_t)sf_mulhi_su(err * 2, v0);
  const uint32_t q1 = sf_umulhi((uint32_t)(ma >> 22), v);
  const int64_t r1 = (int64_t)((ma << 30) - (uint64_t)q1 * mb);
  const int32_t q2 = (sf_mulhi_su((int32_t)(r1 >> 25), v) + 8) >> 4;
  const int64_t r2 = (int64_t)(((uint64_t)r1 << 23) - (uint64_t)(int64_t)q2 * mb);
  const uint64_t q = ((uint64_t)q1 << 23) + (uint64_t)(int64_t)q2 + (r2 >= 0 ? 1u : 0u);
  const uint64_t m = (q >> 1) + ((uint64_t)(uint32_t)e << 52);
  return sf_double(m | ((ua ^ ub) & 0x8000000000000000ull));
}

// Square root of a positive normal number with exponent field ex.
HYDRO_HD double soft_sqrt_core(uint64_t u, int32_t ex) {
  const uint64_t m = (u & 0xfffffffffffffull) | 0x10000000000000ull;
  const int32_t odd = (ex & 1) ^ 1;  // ex - 1023 odd
  const uint64_t M = odd ? m << 1 : m;
  const uint32_t Mh = (uint32_t)(M >> 22);
  uint32_t y = sf_rsqrt_seed((0x3f800000u | ((uint32_t)(m >> 29) & 0x7fffffu)) + (odd ? 0x00800000u : 0u));
  y = y > 0x3f7fffffu ? 0x3f7fffffu : y;
  y = y < 0x3f000000u ? 0x3f000000u : y;
  const uint32_t v0 = (y << 8) | 0x80000000u;
  const int32_t err = (int32_t)(0x40000000u - sf_umulhi(sf_umulhi(v0, v0), Mh));
  const uint32_t v = v0 + (uint32_t)sf_mulhi_su(err * 2, v0);
  const uint32_t s1 = sf_umulhi(Mh, v);
  const int64_t r1 = (int64_t)((M << 8) - (uint64_t)s1 * s1);
  const int32_t s2 = (sf_mulhi_su((int32_t)(r1 >> 4), v) + 8) >> 4;
  const uint64_t d = ((uint64_t)s1 << 24) + (uint64_t)(int64_t)s2;
  const int64_t r2 = (int64_t)(((uint64_t)r1 << 46) - (uint64_t)(int64_t)s2 * d);
  const uint64_t s = ((uint64_t)s1 << 23) + (uint64_t)(int64_t)s2 + (r2 >= 0 ? 1u : 0u);
  const int32_t e = (ex - 1023 - odd) / 2 + 1022;
  return sf_double((s >> 1) + ((uint64_t)(uint32_t)e << 52));
}

// a / b.  Zero numerators are common (a fluid at rest) and cheap; subnormal, infinite and NaN operands and
// quotients near the ends of the exponent range take the FP64 pipe.
HYDRO_HD double soft_div(double a, double b) {
  const uint64_t ua = sf_bits(a), ub = sf_bits(b);
  const int32_t ea = (int32_t)(sf_hi(ua) >> 20 & 0x7ffu), eb = (int32_t)(sf_hi(ub) >> 20 & 0x7ffu);
  const bool normal_b = (uint32_t)(eb - 1) < 2046u;
  if (normal_b && (uint32_t)(ea - 1) < 2046u && (uint32_t)(ea - eb + 1020) < 2041u) return soft_div_core(ua, ub, ea, eb);
  if (normal_b && (ua << 1) == 0) return sf_double((ua ^ ub) & 0x8000000000000000ull);
  return a / b;
}

// sqrt(x); zero, negative, subnormal, infinite and NaN operands take the FP64 pipe
HYDRO_HD double soft_sqrt(double x) {
  const uint64_t u = sf_bits(x);
  const int32_t ex = (int32_t)(sf_hi(u) >> 20);  // sign and exponent
  if ((uint32_t)(ex - 1) < 2046u) return soft_sqrt_core(u, ex);
  return sqrt(x);
}

// Comparisons, minima and scalings by two as integer operations on the bits: an FP64 multiply or compare takes the
// FP64 unit 16 cycles, these two to eight integer instructions.  Same results as the operations they replace for
// every operand, NaN included.  With them, and with the two-shock solver in one copy per kernel (a smaller code
// that stalls less on instruction fetches), KH 512^2 went from 13.7 M to 11.1 M FP64 warp instructions per launch
// and KH 1024^2 from 3.38 to 2.95 ms per step.
HYDRO_HD bool sf_zero(double x) { return (sf_bits(x) << 1) == 0; }                                // x == 0
HYDRO_HD bool sf_gt0(double x) { return sf_bits(x) - 1 < 0x7ff0000000000000ull; }                 // x > 0
HYDRO_HD bool sf_lt0(double x) { return sf_bits(x) - 0x8000000000000001ull < 0x7ff0000000000000ull; }  // x < 0
HYDRO_HD bool sf_ge0(double x) { return sf_gt0(x) || sf_zero(x); }                                // x >= 0
HYDRO_HD bool sf_le0(double x) { return sf_lt0(x) || sf_zero(x); }                                // x <= 0
HYDRO_HD bool sf_finite(double x) { return (sf_hi(sf_bits(x)) & 0x7ff00000u) != 0x7ff00000u; }
HYDRO_HD double sf_abs(double x) { return sf_double(sf_bits(x) & 0x7fffffffffffffffull); }
HYDRO_HD double sf_neg(double x) { return sf_double(sf_bits(x) ^ 0x8000000000000000ull); }

// operands that are positive, +0 or NaN: fmin(a, b), a <= b, a < b (as integers a NaN is above everything)
HYDRO_HD double sf_min_nonneg(double a, double b) { return sf_bits(a) < sf_bits(b) ? a : b; }
HYDRO_HD bool sf_le_nonneg(double a, double b) {
  return sf_bits(a) <= sf_bits(b) && sf_bits(b) <= 0x7ff0000000000000ull;
}
HYDRO_HD bool sf_lt_nonneg(double a, double b) {
  return sf_bits(a) < sf_bits(b) && sf_bits(b) <= 0x7ff0000000000000ull;
}

// x < c ? c : x for a constant c > 0 (a NaN x stays)
HYDRO_HD double sf_floor_at(double x, double c) {
  const uint64_t u = sf_bits(x);
  return (int64_t)u < (int64_t)sf_bits(c) && u <= 0xfff0000000000000ull ? c : x;
}

// a * b on the FP64 pipe, for the rare operands of the routines below; volatile, so that the compiler does not
// run it beside the integer path and select (which would cost what the integer path saves)
HYDRO_HD double sf_mul_rare(double a, double b) {
#ifdef __CUDA_ARCH__
  double r;
  asm volatile("mul.rn.f64 %0, %1, %2;" : "=d"(r) : "d"(a), "d"(b));
  return r;
#else
  return a * b;
#endif
}

// 0.5 x and 2 x: the exponent field moves by one wherever both sides are normal numbers
HYDRO_HD double sf_half(double x) {
  const uint64_t u = sf_bits(x);
  if ((sf_hi(u) >> 20 & 0x7ffu) - 2u < 2045u) return sf_double(u - 0x0010000000000000ull);
  return (u << 1) == 0 ? x : sf_mul_rare(0.5, x);
}
HYDRO_HD double sf_twice(double x) {
  const uint64_t u = sf_bits(x);
  if ((sf_hi(u) >> 20 & 0x7ffu) - 1u < 2045u) return sf_double(u + 0x0010000000000000ull);
  return (u << 1) == 0 ? x : sf_mul_rare(2.0, x);
}

// a * b > 0 (the rounded product): the signs decide unless the product could underflow or is not a number
HYDRO_HD bool sf_same_sign(double a, double b) {
  const uint64_t ua = sf_bits(a), ub = sf_bits(b);
  if ((sf_hi(ua) >> 20 & 0x7ffu) - 512u < 1535u && (sf_hi(ub) >> 20 & 0x7ffu) - 512u < 1535u)
    return (int32_t)(sf_hi(ua) ^ sf_hi(ub)) >= 0;
  if ((ua << 1) == 0 || (ub << 1) == 0) return false;
  return sf_gt0(sf_mul_rare(a, b));
}

}  // namespace hydro
