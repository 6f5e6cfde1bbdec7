// Device-side definitions shared by the library's kernels and by the kernels
// the library generates and compiles at run time for a loaded mechanism
// (runtime compilation has no C++ standard headers: the few types and macros
// used are provided here).  Mechanism blob: one contiguous FP64 array holding
// the species and reaction data of a mechanism (Sec. 2.3 eq. (reaction):
// nu'_{aj}, nu''_{aj}; Arrhenius K_f; third-body efficiencies; Troe falloff;
// NASA-7 thermo).  The same bytes live in device memory and are staged into
// shared memory by the kernels, so every record has a fixed size and an 8-byte
// alignment.
#pragma once
#ifdef __CUDACC_RTC__
typedef unsigned char uint8_t;
typedef int int32_t;
typedef unsigned int uint32_t;
typedef long long int64_t;
typedef unsigned long long uint64_t;
#ifndef INFINITY
#define INFINITY __longlong_as_double(0x7ff0000000000000ULL)
#endif
#ifndef NAN
#define NAN __longlong_as_double(0x7ff8000000000000ULL)
#endif
// per-cell status codes (the values of include/df_chem.h)
#define DF_CELL_OK 0
#define DF_CELL_MAXSTEPS 1
#define DF_CELL_NONFINITE 2
#define DF_CELL_HMIN 3
#else
#include <cmath>
#include <cstdint>
#include <cstring>

#include "../../include/df_chem.h"
#endif

namespace df {

// physical constants (cgs inside the kernels)
constexpr double RU = 8.314462618e7;         // erg/(mol K)
constexpr double RU_SI = 8.314462618;        // J/(mol K)
constexpr double P_STD = 1.01325e6;          // standard-state pressure, dyn/cm^2
constexpr double LN10 = 2.302585092994045684;
constexpr double LOG_PSTD_RU = -4.4074185890025275;     // ln(P_STD / RU), RU in erg/(mol K)

constexpr int MAX_SPECIES = 64;
constexpr int MAX_REACTIONS = 4096;
constexpr int THREAD_PATH_MAX_N = 16;   // N <= this runs one cell per thread

// --- blob layout (all in doubles) -----------------------------------------
// species record k (SP_REC doubles):   W, 1/W, a1..a7, then the NASA-7
//   coefficients as the enthalpy and entropy polynomials use them:
//   a2/2, a3/3, a4/4, a5/5 (h/RT) and a3/2, a4/3, a5/4 (s/R)
constexpr int SP_REC = 16;
constexpr int SP_H = 9;   // offset of a2/2 .. a5/5
constexpr int SP_S = 13;  // offset of a3/2 .. a5/4
// reaction record j (RX_REC doubles):  lnA, beta, Ea/R, meta0, meta1
//   meta0 (8 bytes): reac[3], prod[3] species indices, nr | np << 4, flags
//     flags: bit0-1 type (0 elementary, 1 third-body, 2 Troe), bit2 reversible
//   meta1 (8 bytes): int32 effslot (-1: none), int32 troeslot (-1: none)
constexpr int RX_REC = 5;
// Troe record (TR_REC doubles): lnA0 - lnA, beta0, Ea0/R, alpha, 1/T***, 1/T*, T**, pad
constexpr int TR_REC = 8;
// efficiency record: N doubles per third-body / falloff reaction
// then, past the total (never staged into shared memory), the 64-bit words of the
// fixed-point rate arguments (FixLayout)

struct RxMeta {
  uint8_t reac[3];
  uint8_t prod[3];
  uint8_t nrnp;
  uint8_t flags;
};
static_assert(sizeof(RxMeta) == 8, "meta layout");
struct RxSlots {
  int32_t eff;
  int32_t troe;
};
static_assert(sizeof(RxSlots) == 8, "slot layout");

struct MechDims {
  int N, M, n_eff, n_troe;
  int off_sp, off_rx, off_tr, off_eff, total;  // offsets in doubles
  __host__ __device__ int off_fix() const { return total; }
  __host__ __device__ int allocated() const;
};

// The words behind the blob, all values times log2(e) unless noted:
//   lnA     M      ln A_j 2^53, or FIX_OFF for a reaction without a rate
//   flag    1      0 if some ln A does not fit (fixed_lnA), 2 if one is FIX_OFF, else 1
//   T_low   1      the lowest temperature the fixed-point arguments cover, as a
//                  double; 0: the mechanism does not fit, nothing below is set
//   g       7 N    g_k/RT: the constant 2^53, then the signed coefficients of log2 T
//                  (plain a1, 2^57), T (2^65), T^2 (2^79), T^3 (2^93), T^4 (2^107)
//                  and 1/T (2^46)
//   rate    2 M    b (no log2(e), 2^57) and -E/R (2^46)
//   falloff 3 n_troe  ln A0 - ln A (2^53), b0 - b (2^57), -(E0 - E)/R (2^46)
struct FixLayout {
  int flag, T_low, g, rate, falloff, words;
  __host__ __device__ FixLayout(int N, int M, int n_troe)
      : flag(M), T_low(M + 1), g(M + 2), rate(g + 7 * N), falloff(rate + 2 * M), words(falloff + 3 * n_troe) {}
};
__host__ __device__ inline int MechDims::allocated() const { return total + FixLayout(N, M, n_troe).words; }

inline MechDims mech_dims(int N, int M, int n_eff, int n_troe) {
  MechDims d;
  d.N = N;
  d.M = M;
  d.n_eff = n_eff;
  d.n_troe = n_troe;
  d.off_sp = 0;
  d.off_rx = d.off_sp + SP_REC * N;
  d.off_tr = d.off_rx + RX_REC * M;
  d.off_eff = d.off_tr + TR_REC * n_troe;
  d.total = d.off_eff + n_eff * N;
  return d;
}

#ifdef __CUDACC__
// (double)v for |v| < 2^20, assembled from the integer's sign, leading one and
// the bits below it with integer operations, so that the conversion takes no
// slot of the narrow FP64 pipe (exact: every such integer is a double)
__device__ __forceinline__ double small_int_to_double(int v) {
  const unsigned a = (unsigned)(v < 0 ? -v : v);
  const int lz = __clz(a | 1u);                  // the leading one of a > 0 at bit 31 - lz
  const unsigned mant = ((a << lz) << 1) >> 12;  // the (at most 19) bits below it, left-aligned
  const unsigned hi = ((unsigned)(v < 0) << 31) | ((unsigned)(1023 + 31 - lz) << 20) | mant;
  return __hiloint2double(a != 0u ? (int)hi : 0, 0);
}

// 1/a in FP64 from an FP32 seed and two Newton-Raphson steps r <- r (2 - a r)
// (the relative error squares at each step: 2^-22 -> 2^-44 -> rounding): four
// FP64 operations where a correctly rounded division takes a longer sequence
// on the narrow FP64 pipe.  For |a| inside the FP32 normal range (pivots,
// temperatures, densities, heat capacities, step sizes and error scales of the
// integrators); a zero or non-finite a gives a non-finite result.
__device__ __forceinline__ double rcp_nr(double a) {
  float r0f;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r0f) : "f"((float)a));
  const double r0 = (double)r0f;
  const double r1 = r0 * fma(-a, r0, 2.0);
  return r1 * fma(-a, r1, 2.0);
}

// |a| in [2^-95, 2^97): its FP32 image and that of its reciprocal are normal
__device__ __forceinline__ bool rcp_in_range(double a) {
  return ((uint32_t)__double2hiint(a) & 0x7fffffffu) - 0x3a000000u < 0x46000000u - 0x3a000000u;
}

// 1/a for an a in that range, three FP64 operations: the seed's argument and the
// seed change format through integer operations (a conversion instruction
// occupies the FP64 pipe), the seed's relative error 2^-20 enters cubed
__device__ __forceinline__ double rcp_fast(double a) {
  const uint32_t hi = (uint32_t)__double2hiint(a), sign = hi & 0x80000000u;
  uint32_t r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=r"(r) : "r"(((hi << 3) - 0xc0000000u) | sign));
  const double r0 = __hiloint2double((int)((((r & 0x7fffffffu) >> 3) + 0x38000000u) | sign), (int)(r << 29));
  const double e = fma(-a, r0, 1.0);
  return fma(r0, fma(e, e, e), r0);
}

__device__ __forceinline__ double rcp_any(double a) { return rcp_in_range(a) ? rcp_fast(a) : 1.0 / a; }

#endif

}  // namespace df
