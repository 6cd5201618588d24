// IEEE-754 binary64 division and square root, correctly rounded (to nearest,
// ties to even), on the integer and FP32 pipes.
//
// GB300's FP64 unit is one per SM and serves a warp instruction every 19
// clocks with 64 clocks of latency, whatever the number of active lanes
// (measured).  A division or square root written for it takes about 7.5 such
// slots in a dependent chain: measured 143 SM clocks per warp, 600 clocks of
// latency.  The routines below leave that unit alone: the quotient (root) is
// produced digit by digit in radix 2^20..2^21 -- an FP32 reciprocal (square
// root) from the special-function unit gives each digit from the leading bits
// of an exact 64-bit integer remainder -- and the last remainder's sign makes
// it exact (the schoolbook recurrence; see Knuth, TAOCP vol. 2, 4.3.1 for
// division with estimated digits).  The results are those of the IEEE
// operation, bit for bit.
//
// Measured on the GB300 (clocks per operation, one warp alone / per warp of 32
// on an SM): division 564 / 142 built in, 214 / 22 here; square root 599 / 143
// built in, 254 / 22 here.
//
// Domain of the fast path: normal operands and a result well inside the normal
// range; anything else (zeros, subnormals, infinities, NaN, extreme exponents)
// goes to the built-in operation.
#pragma once

#include <stdint.h>

namespace pic {

__device__ __forceinline__ float fp64i_rcp(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float fp64i_rsqrt(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// rint of the exact a * b for |a * b| < 2^22: the FMA rounds it to an integer
// in the last places of 1.5 * 2^23.
__device__ __forceinline__ int32_t fp64i_digit(float a, float b) {
  return __float_as_int(__fmaf_rn(a, b, 12582912.0f)) - 0x4b400000;
}
// The same for a * b in [0, 2^23), and an exact conversion of |v| < 2^22 (an
// integer addition and an FP32 one; the conversion instruction waits longer).
__device__ __forceinline__ int32_t fp64i_digit_pos(float a, float b) {
  return __float_as_int(__fmaf_rn(a, b, 8388608.0f)) - 0x4b000000;
}
__device__ __forceinline__ float fp64i_float(int32_t v) {
  return __fadd_rn(__int_as_float(v + 0x4b400000), -12582912.0f);
}

// The general operations, out of line: they are the rare path.
static __device__ __noinline__ double fp64i_div_any(double a, double b) { return a / b; }
static __device__ __noinline__ double fp64i_sqrt_any(double a) { return sqrt(a); }

// The significand with its hidden bit, and its top 24 bits as an FP32 number
// in [2^x, 2^(x+1)), x = field - 127 (truncated: up to 2^-23 too small).
__device__ __forceinline__ uint64_t fp64i_sig(uint64_t u) {
  return (u & 0xfffffffffffffull) | 0x10000000000000ull;
}
__device__ __forceinline__ float fp64i_top(uint64_t u, uint32_t field) {
  return __int_as_float((int32_t)(((uint32_t)(u >> 29) & 0x7fffffu) | (field << 23)));
}

// 2^SH a / (B 2^(eb - 1075)) (SH = 0, 1: a power of two does not change the
// rounding), B in [2^52, 2^53], eb in 1 .. 2046, given y =
// (2^52 / B)(1 + e), |e| <= 2^-21.9; neg: the divisor's sign bit in place.
//
// Digits q1 (2^-21), q2 (2^-41), q3 (2^-54) of the significands' quotient A / B
// with exact remainders
//   r1 = 2^21 A - q1 B, |r1| <= 2.4 B (q1's error: y, the truncated A, its own
//   rounding);  r2 = 2^20 r1 - q2 B, |r2| <= 3.3 B (r1 truncated to 22 bits);
//   r3 = 2^13 r2 - q3 B, |r3| <= 0.53 B
// (each fits 64 bits, so it is computed modulo 2^64).  r3 < 0 takes one off:
// Q = floor(2^54 A / B).  A quotient of 53-bit integers is never half-way
// between two 53-bit numbers, so adding half a unit and truncating rounds.
template <int SH>
__device__ __forceinline__ bool fp64i_quot(uint64_t ua, uint64_t B, int eb, float y, uint32_t neg,
                                           double& out) {
  const uint32_t ha = (uint32_t)(ua >> 32);
  const int ea = (int)((ha >> 20) & 0x7ffu);
  const uint64_t A = fp64i_sig(ua);
  const int32_t q1 = fp64i_digit_pos(fp64i_top(ua, 127 + 21), y);
  const uint64_t r1 = (A << 21) - (uint64_t)(uint32_t)q1 * B;
  const int32_t q2 = fp64i_digit(fp64i_float((int32_t)(r1 >> 32) >> 1), __fmul_rn(y, 2.0f));
  const uint64_t r2 = (r1 << 20) - (uint64_t)(int64_t)q2 * B;
  const int32_t q3 = fp64i_digit(fp64i_float((int32_t)(r2 >> 32) >> 1), __fmul_rn(y, 0x1p-6f));
  const uint64_t r3 = (r2 << 13) - (uint64_t)(int64_t)q3 * B;
  const int64_t q12 = ((int64_t)(uint32_t)q1 << 20) + q2;
  const uint64_t Q = (uint64_t)((q12 << 13) + (q3 + ((int32_t)(r3 >> 32) >> 31)));
  const bool big = (Q >> 54) != 0;  // A >= B
  const uint64_t mant = big ? (Q + 2) >> 2 : (Q + 1) >> 1;
  const int de = ea - eb + (1022 + SH) - (big ? 0 : 1);  // exponent field less one (the hidden bit adds it)
  const uint64_t sign = (uint64_t)((ha ^ neg) & 0x80000000u) << 32;
  // the dividend normal, the result's exponent field in 1 .. 2044; zero is
  // common (no field ahead of the wave's front)
  const bool zero = (ua << 1) == 0;
  out = __longlong_as_double((long long)(zero ? sign : (mant + ((uint64_t)(uint32_t)de << 52)) | sign));
  return zero || ((unsigned)(ea - 1) < 2046u && (unsigned)de < 2044u);
}

__device__ __forceinline__ double div_rn(double a, double b) {
  const uint64_t ub = (uint64_t)__double_as_longlong(b);
  const uint32_t hb = (uint32_t)(ub >> 32);
  const int eb = (int)((hb >> 20) & 0x7ffu);
  double q;
  const bool ok = fp64i_quot<0>((uint64_t)__double_as_longlong(a), fp64i_sig(ub), eb,
                                fp64i_rcp(fp64i_top(ub, 127)), hb, q);
  return ok && (unsigned)(eb - 1) < 2046u ? q : fp64i_div_any(a, b);
}

// The rounded significand (53 bits, or 2^53) of sqrt(a), its exponent field
// (for a significand below 2^53) and y = 1 / (significand / 2^52) to 2^-22;
// false for anything but a positive normal a.
//
// m = the significand (times 2 for an odd exponent), s^2 = m / 2^52 in [1, 4);
// y = (1/s)(1 + e), |e| <= 2^-22.4.  Digits s1 (2^-21), s2 (2^-41), s3 (2^-53)
// of s with exact remainders
//   r1 = m - 2^10 s1^2, |r1| < 2^34;  r2 = 2^30 m - t2^2, t2 = 2^20 s1 + s2,
//   |r2| < 2^44.5;  r3 = 2^54 m - T^2, T = 2^12 t2 + s3, |r3| < 2^54.2
// (modulo 2^64).  r3 < 0 takes one off: T = floor(2^53 s); 2^54 m is even, so
// an odd T is never exact and adding one and halving rounds.
__device__ __forceinline__ bool fp64i_sqrt(double a, uint64_t& sig, int& field, float& y) {
  const uint64_t ua = (uint64_t)__double_as_longlong(a);
  const int e = (int)((uint32_t)(ua >> 32) >> 20);  // with the sign: a negative one is out of range
  const uint32_t odd = (e & 1) ^ 1;  // e - 1023 odd
  const uint64_t m = fp64i_sig(ua) << odd;
  y = fp64i_rsqrt(fp64i_top(ua, 127 + odd));
  const int32_t s1 = fp64i_digit_pos(fp64i_top(ua, 127 + 21 + odd), y);
  const uint64_t r1 = m - (((uint64_t)(uint32_t)s1 * (uint32_t)s1) << 10);
  const int32_t s2 = fp64i_digit(fp64i_float((int32_t)(r1 >> 12)), y);
  const uint64_t r2 = (r1 << 30) - ((uint64_t)((int64_t)s1 * s2) << 21) - (uint64_t)((int64_t)s2 * s2);
  const int32_t s3 = fp64i_digit(fp64i_float((int32_t)(r2 >> 23)), __fmul_rn(y, 0x1p-7f));
  const int64_t t2 = ((int64_t)s1 << 20) + s2;
  const uint64_t r3 = (r2 << 24) - (((uint64_t)t2 * (uint64_t)(int64_t)s3) << 13) - (uint64_t)((int64_t)s3 * s3);
  const uint64_t T = (uint64_t)((t2 << 12) + (s3 + ((int32_t)(r3 >> 32) >> 31)));
  sig = (T + 1) >> 1;
  field = (e + 1023) >> 1;
  return (unsigned)(e - 1) < 2046u;
}
__device__ __forceinline__ double fp64i_pack(uint64_t sig, int field) {
  return __longlong_as_double((long long)(sig + ((uint64_t)(uint32_t)(field - 1) << 52)));
}

__device__ __forceinline__ double sqrt_rn(double a) {
  uint64_t sig;
  int field;
  float y;
  return fp64i_sqrt(a, sig, field, y) ? fp64i_pack(sig, field) : fp64i_sqrt_any(a);
}

// The same without branches, for a caller that strings several together and
// looks at the result's validity once (false: an operand or a result outside
// the domain, the values are to be ignored): 2 a / b rounded once (also where 2 a
// would overflow: the push's b = 1 + a^2 is then infinite, outside the domain);
// and g = sqrt(a) with
// t / g (TWO: and u / g), which start from the root's own reciprocal.
__device__ __forceinline__ bool div2_try(double a, double b, double& q) {
  const uint64_t ub = (uint64_t)__double_as_longlong(b);
  const uint32_t hb = (uint32_t)(ub >> 32);
  const int eb = (int)((hb >> 20) & 0x7ffu);
  return fp64i_quot<1>((uint64_t)__double_as_longlong(a), fp64i_sig(ub), eb, fp64i_rcp(fp64i_top(ub, 127)),
                       hb, q) &
         ((unsigned)(eb - 1) < 2046u);
}
template <bool TWO>
__device__ __forceinline__ bool div_sqrt_try(double t, double u, double a, double& qt, double& qu, double& g) {
  uint64_t sig;
  int field;
  float y;
  bool ok = fp64i_sqrt(a, sig, field, y);
  g = fp64i_pack(sig, field);
  if constexpr (TWO) ok &= fp64i_quot<0>((uint64_t)__double_as_longlong(u), sig, field, y, 0u, qu);
  return ok & fp64i_quot<0>((uint64_t)__double_as_longlong(t), sig, field, y, 0u, qt);
}

}  // namespace pic
