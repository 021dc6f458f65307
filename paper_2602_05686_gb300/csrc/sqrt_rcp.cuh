// Square root and reciprocal of a Cholesky pivot in integer arithmetic.
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

namespace sa {

__host__ __device__ __forceinline__ uint64_t mul_hi64(uint64_t a, uint64_t b) {
#ifdef __CUDA_ARCH__
  return __umul64hi(a, b);
#else
  return (uint64_t)(((unsigned __int128)a * b) >> 64);
#endif
}
__host__ __device__ __forceinline__ uint64_t f64_bits(double d) {
#ifdef __CUDA_ARCH__
  return (uint64_t)__double_as_longlong(d);
#else
  uint64_t b;
  memcpy(&b, &d, 8);
  return b;
#endif
}
__host__ __device__ __forceinline__ double f64_of(uint64_t b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double d;
  memcpy(&d, &b, 8);
  return d;
#endif
}

// s = sqrt(d) and r = 1 / s, both rounded to nearest, for a positive normal d
// (its bits), from yb, the bits of an FP32 approximation of 1 / sqrt(mu), mu = d
// scaled by an even power of two into [1, 4): Newton's iteration for the
// reciprocal square root of the significand in fixed point (two steps: 2^-60),
// then the integer square root and quotient settled by their exact remainders
// (taken modulo 2^64, where they fit).  No FP64 instruction: a dependent one
// takes 65 cycles here, and this pair is the chain of a Cholesky pivot (574
// cycles, 954 as sqrt() and a divide).  Equal to sqrt() and 1.0 / s with an
// approximation up to four units off (tests: on the host and on the GPU).
__host__ __device__ __forceinline__ void sqrt_rcp_from(uint64_t db, uint32_t yb, double& s, double& r) {
  // d = m 2^p, p even, m in [2^52, 2^54); mu = m 2^-52 in [1, 4)
  uint64_t m = (db & 0xfffffffffffffull) | 0x10000000000000ull;
  int p = (int)(db >> 52) - 1075;
  const int odd = p & 1;
  m <<= odd;
  p -= odd;
  // y in [0.5, 1] as Q0.32
  uint32_t y0 = yb >= 0x3f800000u ? 0xffffffffu : (((yb & 0x7fffff) | 0x800000) << 8);
  if (yb < 0x3f000000u) y0 = 0x80000000u;
  const uint64_t mf = m << 10;  // mu, Q2.62
  uint64_t t = (uint64_t)y0 * y0;
  const int64_t e1 = (int64_t)((1ull << 62) - mul_hi64(mf, t));          // 1 - mu y^2, Q.62
  const uint64_t y1 = ((uint64_t)y0 << 31) + (uint64_t)(((int64_t)(uint64_t)y0 * (int32_t)(e1 >> 12)) >> 20);  // Q1.63
  t = mul_hi64(y1, y1);
  const int32_t e2 = (int32_t)((1ull << 60) - mul_hi64(mf, t));          // Q.60
  const uint64_t y2 = y1 + (uint64_t)(((int64_t)(y1 >> 32) * e2) >> 29);
  // S = sqrt(m 2^52) rounded: at most one off before the remainder says so
  uint64_t S = mul_hi64(mf, y2) >> 9;
  int64_t rem = (int64_t)((m << 52) - S * S);
  if (rem < 0) {
    S -= 1;
    rem += (int64_t)(2 * S + 1);
  } else if (rem > (int64_t)(2 * S)) {
    rem -= (int64_t)(2 * S + 1);
    S += 1;
  }
  S += rem > (int64_t)S;
  const int e = (p - 52) / 2;
  s = f64_of(((uint64_t)(e + 1074) << 52) + S);
  // Q = 2^105 / S rounded (no ties: 2^106 has no odd factor)
  uint64_t Q = y2 >> 10;
  int64_t q = (int64_t)(0 - S * Q);
#pragma unroll
  for (int u = 0; u < 2; ++u)
    if (q < 0) {
      Q -= 1;
      q += (int64_t)S;
    }
#pragma unroll
  for (int u = 0; u < 2; ++u)
    if (q >= (int64_t)S) {
      Q += 1;
      q -= (int64_t)S;
    }
  Q += 2 * q > (int64_t)S;
  r = f64_of(((uint64_t)(969 - e) << 52) + Q);
}

// mu of sqrt_rcp_from to 23 bits
__host__ __device__ __forceinline__ uint32_t rsqrt_arg(uint64_t db) {
  const uint32_t hi = (uint32_t)(db >> 32), lo = (uint32_t)db;
  const uint32_t odd = ((hi >> 20) - 1075) & 1;
  return ((127 + odd) << 23) | ((hi & 0xfffff) << 3) | (lo >> 29);
}

__device__ __forceinline__ void sqrt_rcp(double d, double& s, double& r) {
  const uint64_t db = f64_bits(d);
  const int ex = (int)(db >> 52);
  if (ex == 0 || ex >= 2047) {  // zero exponent, infinity, NaN, negative
    s = sqrt(d);
    r = 1.0 / s;
    return;
  }
  float yf;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(yf) : "f"(__int_as_float((int)rsqrt_arg(db))));
  sqrt_rcp_from(db, (uint32_t)__float_as_int(yf), s, r);
}

}  // namespace sa
