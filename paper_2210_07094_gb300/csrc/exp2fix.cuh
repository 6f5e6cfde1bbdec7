// exp(x) and 2^x in 64-bit fixed point on the integer pipes.
//
// The FP64 pipe issues one warp instruction in 64 cycles; a 32 x 32 -> 64 bit
// multiply-add takes 4 and an addition 1.  The table-driven exponential of
// fastexp.cuh is 8 FP64 instructions, 670 cycles per warp; the one below is
// about 60 integer instructions: 161 cycles alone on a sub-partition, 115 with
// several warps (152 SMs, dependent chains of two).  Its argument reduction is
// exact but for one rounding, so it is also the more accurate: at most 0.93 ulp
// for |x| <= 128 and 1.08 for |x| < 512, against 1.32 (host emulation, 3e6
// arguments per range).
//
// X = x 2^53 in a 64-bit integer, |x| < 1022: m = X >> 53, j = the next 8 bits,
// g = the 45 bits below them as a fraction of 2^-8:
//   2^x = 2^m 2^(j/256) (1 + p),  p = g (a1 + g (a2 + g (a3 + g a4)))
// with 2^(j/256) a 64-bit fraction from a 2 KB table.  The table is read from
// global memory through L1: a gather of 8-byte entries costs there what it
// costs in shared memory (112 against 115 cycles per exponential), and the
// shared memory stays free for cells.
#pragma once
#include "dev_common.cuh"

namespace df {

#include "exp2fix_table.inc"

__host__ __device__ __forceinline__ uint64_t wmad(uint32_t a, uint32_t b, uint64_t c) { return (uint64_t)a * b + c; }

// the high 64 bits of a 64 x 64 bit product to within 3 units (the product of
// the low words and the carries out of the cross products' low words dropped)
__device__ __forceinline__ uint64_t mulhi64_3(uint32_t ah, uint32_t al, uint32_t bh, uint32_t bl) {
  return wmad(ah, bh, (uint64_t)__umulhi(ah, bl)) + __umulhi(al, bh);
}

// 2^((X + 1/2) 2^-53) = r 2^(e - 63) with r in [2^63, 2^64): X is the floor of a
// value, its mean the half unit above
__device__ __forceinline__ uint64_t exp2_parts(int64_t X, int& e) {
  const uint32_t xh = (uint32_t)((uint64_t)X >> 32), xl = (uint32_t)X;
  const uint64_t t = __ldg(reinterpret_cast<const unsigned long long*>(g_exp2fix_tab) + ((xh >> 13) & 255u));
  const uint32_t gh = (xh << 19) | (xl >> 13), gl = (xl << 19) | (1u << 18);
  const uint32_t h3 = (uint32_t)EXP2FIX_A3 + __umulhi(gh, (uint32_t)EXP2FIX_A4);  // 2^60
  const uint64_t h2 = wmad(__umulhi(gh, h3), 1u << 22, EXP2FIX_A2);              // 2^82
  const uint64_t h1 = EXP2FIX_A1 + (mulhi64_3(gh, gl, (uint32_t)(h2 >> 32), (uint32_t)h2) >> 10);  // 2^72
  const uint64_t p = mulhi64_3(gh, gl, (uint32_t)(h1 >> 32), (uint32_t)h1);                       // 2^72
  const uint64_t q = mulhi64_3((uint32_t)(t >> 32), (uint32_t)t, (uint32_t)(p >> 32), (uint32_t)p);
  e = (int32_t)xh >> 21;
  return t + (q >> 8);
}

// the same as a double, |X| < 1022 2^53 (normal results): the leading 53 bits,
// rounded; the leading one adds 1 to the exponent field
__device__ __forceinline__ double exp2_fixed(int64_t X) {
  int e;
  const uint64_t r = exp2_parts(X, e);
  const uint64_t f = (uint64_t)((uint32_t)(e + 1022) << 20) << 32;
  return __longlong_as_double((long long)(f + (r >> 11) + ((r >> 10) & 1u)));
}

// Rates as unpacked floating-point numbers m 2^e: a product of a rate constant
// with up to three concentrations is a chain of integer multiplications, seven
// instructions each where an FP64 multiplication occupies its pipe for 64 cycles.
// The constant enters with 64 bits, each concentration with 53 at bit 62, and a
// product drops at most two leading bits, so 57 remain after three.  Packing truncates
// to 53, towards zero by up to one unit in the last place, where an FP64 product rounds
// at each multiplication, by half a unit.  The sign is the top bit of the concentrations'
// exclusive or, carried beside.
struct Fx {
  uint64_t m;
  int e;
};

// a finite double for fx_mul (e: the exponent's share of the product); zeros and
// subnormals become numbers that pack to zero
__device__ __forceinline__ Fx fx_factor(double x) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x), e = (hi >> 20) & 0x7ffu;
  Fx a;
  a.m = ((uint64_t)(0x40000000u | ((hi << 10) & 0x3fffffffu) | (lo >> 22)) << 32) | (lo << 10);
  a.e = e ? (int)e - 1021 : -100000;
  return a;
}

__device__ __forceinline__ Fx fx_mul(Fx a, Fx c) {
  Fx p;
  p.m = mulhi64_3((uint32_t)(a.m >> 32), (uint32_t)a.m, (uint32_t)(c.m >> 32), (uint32_t)c.m);
  p.e = a.e + c.e;
  return p;
}

// sign m 2^e as a double (truncated), 0 below the normal range, infinity above it
__device__ __forceinline__ double fx_pack(uint64_t m, int e, uint32_t sign) {
  const int lz = __clzll((long long)m);
  const uint64_t r = m << (lz & 63);
  const uint32_t f = (uint32_t)(e - lz + 1085);  // exponent field - 1
  uint64_t b = ((uint64_t)(f << 20) << 32) + (r >> 11);
  if (f >= 2046u || m == 0) b = (int)f < 0 || m == 0 ? 0 : 0x7ff0000000000000ull;
  return __longlong_as_double((long long)(b | ((uint64_t)(sign & 0x80000000u) << 32)));
}
__device__ __forceinline__ double fx_pack(Fx a, uint32_t sign) { return fx_pack(a.m, a.e, sign); }

// a - b, signs apart; both m below 2^63
__device__ __forceinline__ double fx_diff(Fx a, uint32_t sa, Fx b, uint32_t sb) {
  const int d = a.e - b.e;
  const uint64_t am = a.m >> min(max(-d, 0) + 1, 63), bm = b.m >> min(max(d, 0) + 1, 63);
  const int64_t opp = (int64_t)((int32_t)(sa ^ sb) >> 31);  // all ones: the magnitudes add
  const int64_t v = (int64_t)am - (((int64_t)bm ^ opp) - opp);
  const int64_t neg = v >> 63;
  return fx_pack((uint64_t)((v ^ neg) - neg), max(a.e, b.e) + 1, sa ^ (uint32_t)(neg >> 32));
}

// 2^((X + 1/2) 2^-53) of n exponents in a vector of 64-bit words, in place, |X| <
// 1022 2^53: the leading 53 bits and the exponent (e + 1024) in the low 11.  Four
// at a time, independent chains in one loop body: a warp alone on its
// sub-partition waits out the latency of each dependent integer instruction
// otherwise, and the code is there once.
template <int N, class V>
__device__ __forceinline__ void fx_exp2_all(V S) {
#pragma unroll 1
  for (int i = 0; i < N; i += 4) {
    uint64_t m[4];
    int e[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) m[k] = exp2_parts(__double_as_longlong(S[i + k]), e[k]);
#pragma unroll
    for (int k = 0; k < 4; ++k)
      S[i + k] = __longlong_as_double((long long)((m[k] & ~0x7ffull) | (uint32_t)((e[k] + 1024) & 0x7ff)));
  }
}

// one of them; the bits the exponent took count as half a unit
__device__ __forceinline__ Fx fx_word(double w) {
  const uint64_t u = (uint64_t)__double_as_longlong(w);
  Fx a;
  a.m = (u & ~0x7ffull) | 0x400u;
  a.e = (int)((uint32_t)u & 0x7ffu) - (1024 + 63);
  return a;
}

// 2^v as a factor for fx_mul, |v| < 1000
__device__ __forceinline__ Fx fx_exp2_factor(double v) {
  const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v), e = (hi >> 20) & 0x7ffu;
  const uint64_t m = ((uint64_t)(0x40000000u | ((hi << 10) & 0x3fffffffu) | (lo >> 22)) << 32) | (lo << 10);
  const uint32_t s = e < 969u ? 63u : 1032u - e;  // floor(|v| 2^53), then the complement
  Fx a;
  a.m = exp2_parts((int64_t)(m >> s) ^ (int64_t)((int32_t)hi >> 31), a.e);
  a.e += 1;
  return a;
}

// v 2^-52 as a double
__device__ __forceinline__ double q52_to_double(int64_t v) {
  const int64_t neg = v >> 63;
  return fx_pack((uint64_t)((v ^ neg) - neg), -52, (uint32_t)(neg >> 32));
}

// v c 2^-64 to within 3 units
__device__ __forceinline__ int64_t mul_fixed_signed(int64_t v, uint64_t c) {
  const int64_t neg = v >> 63;
  const uint64_t a = (uint64_t)((v ^ neg) - neg);
  const uint64_t p = mulhi64_3((uint32_t)(a >> 32), (uint32_t)a, (uint32_t)(c >> 32), (uint32_t)c);
  return ((int64_t)p ^ neg) - neg;
}

// v 2^-bits as a double
__device__ __forceinline__ double fixed_to_double(int64_t v, int bits = 53) {
  const int64_t neg = v >> 63;
  return fx_pack((uint64_t)((v ^ neg) - neg), -bits, (uint32_t)(neg >> 32));
}

// x log2(e) as floor(x log2(e) 2^53), |x| < 512: the 53-bit mantissa (at bit
// 62) times log2(e)/2, shifted by the exponent; a negative x takes the
// complement, so both signs are floors
__host__ __device__ __forceinline__ int64_t exp_arg_fixed(double x) {
  uint64_t bits;
  memcpy(&bits, &x, 8);
  const uint32_t hi = (uint32_t)(bits >> 32), lo = (uint32_t)bits;
  constexpr uint32_t ch = (uint32_t)(EXP2FIX_LOG2E_HALF >> 32), cl = (uint32_t)EXP2FIX_LOG2E_HALF;
  const uint32_t mh = 0x40000000u | ((hi << 10) & 0x3fffffffu) | (lo >> 22), ml = lo << 10;
  const uint64_t p = wmad(mh, ch, wmad(ml, ch, (uint64_t)mh * cl) >> 32);
  const uint32_t e = (hi >> 20) & 0x7ffu;
  const uint32_t s = e < 968u ? 63u : 1031u - e;
  return (int64_t)(p >> s) ^ (int64_t)((int32_t)hi >> 31);
}

// floor(x 2^S) of a positive double whose exponent lets it fit (x 2^S < 2^63)
template <int S>
__device__ __forceinline__ uint64_t pos_fixed(double x) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const uint64_t m = ((uint64_t)(0x40000000u | ((hi << 10) & 0x3fffffffu) | (lo >> 22)) << 32) | (lo << 10);
  return m >> (1085 - S - (int)(hi >> 20));
}

// a b 2^-64 to within 3 units
__device__ __forceinline__ uint64_t mul_fixed(uint64_t a, uint64_t b) {
  return mulhi64_3((uint32_t)(a >> 32), (uint32_t)a, (uint32_t)(b >> 32), (uint32_t)b);
}

// |x| >= 512, inf and NaN (an integer test of the high word)
__device__ __forceinline__ bool exp_is_big(double x) { return (__double2hiint(x) & 0x7fffffff) >= 0x40800000; }

// the fixed-point arguments cover temperatures below this (and from FixLayout.T_low)
constexpr double FIX_T_HIGH = 8000.0;

// the ln A the fixed-point rate arguments are built for (150 octaves): the sums stay
// within what 64 bits hold with what fixed_T_low allows the temperature terms
__host__ __device__ inline bool lnA_fits_fixed(double lnA) { return lnA > -104.0 && lnA < 104.0; }

// The word of a reaction's ln A, false if it does not fit.  A reaction without a rate
// (A = 0, or a falloff reaction whose ln A0 - ln A, d0, is -inf) has one of its own.
constexpr int64_t FIX_OFF = (int64_t)(1ull << 63);
__host__ __device__ inline bool fixed_lnA(double lnA, double d0, int64_t* word) {
  const bool off = lnA == -INFINITY || d0 == -INFINITY, ok = off || lnA_fits_fixed(lnA);
  *word = off ? FIX_OFF : ok ? exp_arg_fixed(lnA) : 0;
  return ok;
}

// x + xc, both within 1022 2^53 and their sum below 1000 2^53, but not below
// -1000 2^53 (a constant of 2^-1000)
__device__ __forceinline__ int64_t add_exponents(int64_t x, int64_t xc) {
  return (x >> 1) + (xc >> 1) < -(500ll << 53) ? -(1000ll << 53) : x + xc;
}

__device__ __forceinline__ double exp_rate(double x) {
  return exp_is_big(x) ? exp(x) : exp2_fixed(exp_arg_fixed(x));
}

// two at once, as one straight-line block (two independent chains); the rare
// big arguments are fixed up afterwards
__device__ __forceinline__ void exp_rate2(double x1, double x2, double& e1, double& e2) {
  const bool b1 = exp_is_big(x1), b2 = exp_is_big(x2);
  e1 = exp2_fixed(exp_arg_fixed(b1 ? 0.0 : x1));
  e2 = exp2_fixed(exp_arg_fixed(b2 ? 0.0 : x2));
  if (b1 | b2) {
    if (b1) e1 = exp(x1);
    if (b2) e2 = exp(x2);
  }
}

}  // namespace df
