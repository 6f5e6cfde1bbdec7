// log2(x) in 64-bit fixed point on the integer pipes (the companion of
// exp2fix.cuh; the same reason: the FP64 pipe issues one warp instruction in 64
// cycles, and a table-driven FP64 logarithm is 13 of them).
//
// x = 2^e y with y in [1, 2); j = the top 8 bits of y's fraction; r_j just above
// 1/(1 + j/256) in 31 bits, so t = y r_j - 1 lies in [0, 2^-8) and its 62-bit
// fraction is exact but for one truncation;
//   log2 x = e - log2 r_j + log2(1 + t),
// log2(1 + t) by a degree-5 polynomial (error below 2^-58).  The sum is good to
// about 2^-57 absolutely: what the rate expressions need, where ln T and the
// log10 of the Troe falloff are addends.
#pragma once
#include "exp2fix.cuh"

namespace df {

#include "log2fix_table.inc"

// log2(y) 2^60 of the mantissa y = 1.f of a double given by its words
__device__ __forceinline__ uint64_t log2_mantissa_fixed(uint32_t hi, uint32_t lo) {
  const Log2FixEntry* t = &g_log2fix_tab[(hi >> 12) & 255u];
  const uint32_t r = __ldg(&t->r);
  const uint64_t l = __ldg(reinterpret_cast<const unsigned long long*>(&t->l));
  const uint32_t mh = 0x80000000u | (hi << 11) | (lo >> 21), ml = lo << 11;
  const uint64_t g = (wmad(mh, r, __umulhi(ml, r)) - (1ull << 62)) << 10;  // t 2^72
  const uint32_t gh = (uint32_t)(g >> 32), gl = (uint32_t)g;
  const uint32_t h4 = (uint32_t)LOG2FIX_B4 - __umulhi(gh, (uint32_t)LOG2FIX_B5);
  const uint32_t h3 = (uint32_t)LOG2FIX_B3 - (__umulhi(gh, h4) >> 8);
  const uint64_t h2 = LOG2FIX_B2 - (wmad(gh, h3, 0) >> 9);
  const uint64_t h1 = LOG2FIX_B1 - (mulhi64_3(gh, gl, (uint32_t)(h2 >> 32), (uint32_t)h2) >> 9);
  return l + (mulhi64_3(gh, gl, (uint32_t)(h1 >> 32), (uint32_t)h1) >> 11);
}

// log2(x) 2^60 for 1 <= x < 2^15
__device__ __forceinline__ uint64_t log2_fixed(double x) {
  const uint32_t hi = (uint32_t)__double2hiint(x);
  return ((uint64_t)((hi >> 20) - 1023u) << 60) + log2_mantissa_fixed(hi, (uint32_t)__double2loint(x));
}

// log2(x) 2^52 of a normal positive double
__device__ __forceinline__ int64_t log2_q52(double x) {
  const int hi = __double2hiint(x);
  return ((int64_t)((hi >> 20) - 1023) << 52) +
         (int64_t)((log2_mantissa_fixed((uint32_t)hi, (uint32_t)__double2loint(x)) + 128u) >> 8);
}

// ln(x) log_b(e) for any x; hi + lo = ln 2 log_b(e) with hi rounded to 42 bits, so
// that a multiple of it by the exponent is exact.  Zero, negative, subnormal,
// infinite and NaN arguments go to the library's log.  Four FP64 operations.
__device__ __forceinline__ double log_scaled(double x, double hi, double lo, double logb_e) {
  const int xh = __double2hiint(x);
  if (xh < 0x00100000 || xh >= 0x7ff00000) return log(x) * logb_e;
  // the fraction as 1.f - 1 (exact), the exponent through integer operations
  const uint64_t m = log2_mantissa_fixed((uint32_t)xh, (uint32_t)__double2loint(x));
  const double f = __longlong_as_double((long long)(0x3ff0000000000000ull + ((m + 128u) >> 8))) - 1.0;
  const double e = small_int_to_double((xh >> 20) - 1023);
  return fma(e, hi, fma(e, lo, f * (hi + lo)));
}

__device__ __forceinline__ double log_rate(double x) {
  return log_scaled(x, 0x1.62e42fefa3800p-1, 0x1.ef35793c76730p-45, 1.0);
}
__device__ __forceinline__ double log10_rate(double x) {
  return log_scaled(x, 0x1.34413509f7800p-2, 0x1.fef311f12b358p-46, 0.43429448190325182765);
}

}  // namespace df
