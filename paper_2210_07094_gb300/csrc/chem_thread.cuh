// Device chemistry for the one-cell-per-thread path (N <= 16 species).
//
// Per-thread vectors whose index is a compile-time constant live in registers;
// vectors indexed by a reaction's species (C, wdot, g/RT, h/RT) and the dense
// (N+1)x(N+1) Jacobian / LU live in shared memory in [index][thread] order, so
// that the 32 lanes of a warp touch 32 consecutive doubles (no bank conflicts).
//
// Equations (cgs units inside):
//   rho = p W/(R T),  C_k = rho Y_k / W_k                        (Sec. 2.3)
//   K_f = A T^b exp(-Ea/RT)  (Arrhenius law, Sec. 2.3)
//   K_r = K_f / K_c,  K_c = exp(-sum_k nu_kj g_k/RT) (p_std/RT)^{sum_k nu_kj}
//   third body: rate x [M], [M] = sum_k eps_k C_k
//   Troe: k = k_inf Pr/(1+Pr) F, Pr = k_0 [M]/k_inf,
//         log F = log F_c / (1 + ((log Pr + c)/(n - d (log Pr + c)))^2)
//   q_j = K_f prod C^nu' - K_r prod C^nu''
//   dY_k/dt = W_k sum_j (nu''_kj - nu'_kj) q_j / rho           (eq. (sourceeq))
//   dT/dt = -sum_k H_k wdot_k / (rho cp)   (constant-pressure adiabatic 0D reactor,
//                                           Sec. 2.2 df0DFoam; h conserved)
#pragma once
#include "dev_common.cuh"
#include "dual.cuh"
#include "log2fix.cuh"

namespace df {

// ln and log10 of the rate expressions by the fixed-point logarithm (the
// dual-number version carries the derivative d/x)
__device__ __forceinline__ double fast_log(double x) { return log_rate(x); }
__device__ __forceinline__ double fast_log10(double x) { return log10_rate(x); }
__device__ __forceinline__ Dual fast_log10(const Dual& x) {
  return Dual(log10_rate(x.v), x.d / (x.v * 2.302585092994045684));
}

// strided view of a per-thread vector (any scalar type) in shared memory; a
// stride fixed at compile time (ST > 0, the block size) turns the address of
// every constant index into an immediate offset
template <class S, int ST = 0>
struct SVT {
  S* p;
  int s;
  __device__ __forceinline__ S& operator[](int i) const { return p[i * (ST > 0 ? ST : s)]; }
};
typedef SVT<double> SV;

struct MechView {
  const double* sp;
  const double* rx;
  const double* tr;
  const double* eff;
  const long long* fix;  // the fixed-point words (FixLayout), always in global memory
  int M;
  int fg, fr, ff;        // offsets of their species, reaction and falloff records
  double T_low;          // the fixed-point arguments cover T_low <= T < FIX_T_HIGH; infinity: none
};

// blob: the mechanism as the kernel reads it (shared or global memory); global: in
// global memory, with the words behind it
__device__ __forceinline__ MechView make_view(const double* blob, const MechDims& d, const double* global) {
  MechView v;
  v.sp = blob + d.off_sp;
  v.rx = blob + d.off_rx;
  v.tr = blob + d.off_tr;
  v.eff = blob + d.off_eff;
  v.M = d.M;
  const FixLayout F(d.N, d.M, d.n_troe);
  v.fix = reinterpret_cast<const long long*>(global + d.off_fix());
  v.fg = F.g;
  v.fr = F.rate;
  v.ff = F.falloff;
  v.T_low = __longlong_as_double(v.fix[F.T_low]);
  // with a reaction without a rate in FP64: a test for one in rate_fixed made every
  // mechanism 1 to 5% slower (constant volume 20011 cells 4.77 -> 4.84 ms, 8192 cells of 50 species
  // 119.9 -> 122.1, 16411 source terms 64 -> 68 us) and such a one 13% faster
  if (!(v.T_low > 0.0) || v.fix[F.flag] != 1) v.T_low = INFINITY;
  return v;
}

__device__ __forceinline__ RxMeta load_meta(const double* r) {
  RxMeta m;
  unsigned long long bits = __double_as_longlong(r[3]);
  memcpy(&m, &bits, 8);
  return m;
}
__device__ __forceinline__ RxSlots load_slots(const double* r) {
  RxSlots s;
  unsigned long long bits = __double_as_longlong(r[4]);
  memcpy(&s, &bits, 8);
  return s;
}

// exp of two arguments (two independent dependency chains for the scheduler)
__device__ __forceinline__ void exp_pair(double a, double b, double& ea, double& eb) { exp_rate2(a, b, ea, eb); }
__device__ __forceinline__ void exp_pair(const Dual& a, const Dual& b, Dual& ea, Dual& eb) {
  ea = exp_rate(a);
  eb = exp_rate(b);
}

// Result of the rate of one reaction; with J also the pieces of dq/dT|_C and
// dq/dC.
template <class S>
struct RateOutT {
  bool active;
  RxMeta mt;
  RxSlots sl;
  S q;       // net rate [mol/cm^3/s]
  S fk, rk;  // effective forward / reverse coefficients (x [M] for third body)
  S dqdT;    // dq/dT at fixed C
  S dqdM;    // dq/d[M] (third body, Troe); multiplies eps_l for dq/dC_l
  S cr[3], cp[3];
};
typedef RateOutT<double> RateOut;

// Everything rate_one reads from memory for reaction j: its record, the
// concentrations of its species, sum_k nu_kj g_k/RT (and h_k/RT with J) and,
// for a third-body or falloff reaction, [M] = sum_l eps_l C_l.  Gathering the
// next reaction's inputs before the current reaction's production rates are
// stored keeps the shared-memory loads off the FP64 dependency chain (the
// concentrations and g/RT do not change during the reaction loop).
template <class S>
struct RxIn {
  double lnA, beta, EaR;
  RxMeta mt;
  RxSlots sl;
  S cr[3], cp[3];  // reactant / product concentrations (1 where absent)
  S sg, sh;        // sum nu g/RT, sum nu h/RT (products minus reactants)
  S Mc;            // [M] (third body, falloff)
};

// Third-body efficiencies as a sum of all concentrations plus sparse
// corrections: [M] = ctot + sum over the species l whose efficiency is not 1 of
// (eps_l - 1) C_l.  off[s] .. off[s + 1] index the (l, low word, high word)
// triples of efficiency slot s in ent (the correction eps_l - 1 as the two
// 32-bit halves of a double).
struct SparseEff {
  const int* off;
  const int* ent;
  double ctot;
};

template <int NS, bool WITH_J, class S, class Vec>
__device__ __forceinline__ void rate_gather(const MechView& mv, const double* r, int Nrt, const Vec& C,
                                            const Vec& gRT, const Vec& hRT, RxIn<S>& g,
                                            const SparseEff* se = nullptr) {
  const int N = NS > 0 ? NS : Nrt;
  g.lnA = r[0];
  g.beta = r[1];
  g.EaR = r[2];
  g.mt = load_meta(r);
  g.sl = load_slots(r);
  const RxMeta mt = g.mt;
  const int nr = mt.nrnp & 15, np = mt.nrnp >> 4;
  const S one(1.0);
  g.cr[0] = C[mt.reac[0]];
  g.cr[1] = nr > 1 ? S(C[mt.reac[1]]) : one;
  g.cr[2] = nr > 2 ? S(C[mt.reac[2]]) : one;
  g.cp[0] = C[mt.prod[0]];
  g.cp[1] = np > 1 ? S(C[mt.prod[1]]) : one;
  g.cp[2] = np > 2 ? S(C[mt.prod[2]]) : one;
  S sg = gRT[mt.prod[0]] - gRT[mt.reac[0]];
  S sh(0.0);
  if (WITH_J) sh = hRT[mt.prod[0]] - hRT[mt.reac[0]];
  if (np > 1) { sg += gRT[mt.prod[1]]; if (WITH_J) sh += hRT[mt.prod[1]]; }
  if (np > 2) { sg += gRT[mt.prod[2]]; if (WITH_J) sh += hRT[mt.prod[2]]; }
  if (nr > 1) { sg -= gRT[mt.reac[1]]; if (WITH_J) sh -= hRT[mt.reac[1]]; }
  if (nr > 2) { sg -= gRT[mt.reac[2]]; if (WITH_J) sh -= hRT[mt.reac[2]]; }
  g.sg = sg;
  g.sh = sh;
  g.Mc = S(0.0);
  if ((mt.flags & 3) != 0) {
    if (se) {
      S Mc(se->ctot);
      for (int t = se->off[g.sl.eff]; t < se->off[g.sl.eff + 1]; ++t) {
        const int* e = se->ent + 3 * t;
        Mc += __hiloint2double(e[2], e[1]) * C[e[0]];
      }
      g.Mc = Mc;
    } else {
      const double* ef = mv.eff + N * g.sl.eff;
      S Mc(0.0);
#pragma unroll
      for (int l = 0; l < N; ++l) Mc += ef[l] * C[l];
      g.Mc = Mc;
    }
  }
}

// The rate of one reaction from its gathered inputs: Arrhenius K_f, K_r = K_f/K_c,
// third-body [M] and Troe falloff; with WITH_J also dq/dT at fixed C and dq/d[M].
template <int NS, bool WITH_J, class S>
__device__ __forceinline__ void rate_compute(const MechView& mv, const RxIn<S>& g, S T, S lnT, S invT,
                                             S lnP0RT, RateOutT<S>& o) {
  o.active = false;
  const double lnA = g.lnA;
  if (lnA == -INFINITY) return;  // A = 0: no rate
  const double beta = g.beta, EaR = g.EaR;
  const RxMeta mt = g.mt;
  o.mt = mt;
  const int nr = mt.nrnp & 15, np = mt.nrnp >> 4;
  const int type = mt.flags & 3;
  const bool rev = (mt.flags & 4) != 0;
  const S lnkf = lnA + beta * lnT - EaR * invT;
  o.cr[0] = g.cr[0]; o.cr[1] = g.cr[1]; o.cr[2] = g.cr[2];
  o.cp[0] = g.cp[0]; o.cp[1] = g.cp[1]; o.cp[2] = g.cp[2];
  const S Pf = g.cr[0] * g.cr[1] * g.cr[2];
  const S Pb = g.cp[0] * g.cp[1] * g.cp[2];
  const S sg = g.sg, sh = g.sh;
  const int dnu = np - nr;
  // ln(1/K_c); a reaction that keeps its mole count has no pressure term (no
  // operation where the counts are known at compile time, as in the kernels
  // generated for a mechanism; the same value either way)
  const S lnKcinv = dnu == 0 ? sg : sg - (double)dnu * lnP0RT;
  S kf, kr, mult(1.0), dqdM(0.0), dlnk(0.0);
  const RxSlots sl = g.sl;
  o.sl = sl;
  if (type == 2) {
    const double* tr = mv.tr + TR_REC * sl.troe;
    const S Mc = g.Mc;
    const S lnk0 = lnA + tr[0] + tr[1] * lnT - tr[2] * invT;
    // Pr = k0 [M] / kinf, as exp(ln k0 - ln kinf) [M] (no division); the
    // exponentials in pairs (see exp_pair)
    S kinf, r0, e3, e1, e2, invKc;
    exp_pair(lnkf, lnk0 - lnkf, kinf, r0);
    const S Pr = r0 * Mc;
    if (!(val(Pr) > 0.0)) return;  // no low-pressure rate or no collider: k = 0
    exp_pair(-T * tr[4], -T * tr[5], e3, e1);
    exp_pair(-tr[6] * invT, lnKcinv, e2, invKc);
    if (!rev) invKc = S(0.0);
    const S Fc = (1.0 - tr[3]) * e3 + tr[3] * e1 + e2;
    const S Lc = fast_log10(Fc);
    const S cc = -0.4 - 0.67 * Lc;
    const S nn = 0.75 - 1.27 * Lc;
    const S L = fast_log10(Pr);
    const S x = L + cc;
    const S den = nn - 0.14 * x;
    // 1 / (1 + (x / den)^2) with one division
    const S den2 = den * den;
    const S q1 = den2 / (den2 + x * x);
    const S log10F = Lc * q1;
    const S F = exp_rate(LN10 * log10F);
    const S onePr = 1.0 / (1.0 + Pr);
    kf = kinf * Pr * onePr * F;
    kr = kf * invKc;
    if (WITH_J) {
      const S k0 = exp_rate(lnk0);
      const S f1 = x / den;
      const S df1_dL = nn / (den * den);
      const S df1_dLc = (-0.67 * den - x * (-1.27 + 0.67 * 0.14)) / (den * den);
      const S dlogF_dL = -2.0 * Lc * f1 * df1_dL * q1 * q1;
      const S dlogF_dLc = q1 - 2.0 * Lc * f1 * df1_dLc * q1 * q1;
      const S gpr = onePr + dlogF_dL;  // d ln k / d ln Pr
      const S dlnkinf = (beta + EaR * invT) * invT;
      const S dlnk0 = (tr[1] + tr[2] * invT) * invT;
      const S dFc = -(1.0 - tr[3]) * tr[4] * e3 - tr[3] * tr[5] * e1 + tr[6] * invT * invT * e2;
      dlnk = dlnkinf + gpr * (dlnk0 - dlnkinf) + dlogF_dLc * dFc / Fc;
      // dk/d[M] = k0 F gpr / (1 + Pr); rate per unit k is (Pf - Pb/K_c)
      dqdM = k0 * F * gpr * onePr * (Pf - Pb * invKc);
    }
  } else {
    exp_pair(lnkf, lnkf + lnKcinv, kf, kr);
    if (!rev) kr = S(0.0);
    if (type == 1) {
      mult = g.Mc;
      dqdM = kf * Pf - kr * Pb;
    }
    if (WITH_J) dlnk = (beta + EaR * invT) * invT;
  }
  o.active = true;
  o.q = mult * (kf * Pf - kr * Pb);
  o.fk = mult * kf;
  o.rk = mult * kr;
  o.dqdM = dqdM;
  if (WITH_J) {
    const S dlnKc = (sh - (double)dnu) * invT;
    o.dqdT = mult * (kf * Pf * dlnk - kr * Pb * (dlnk - dlnKc));
  } else {
    o.dqdT = S(0.0);
  }
}


// Rate of one reaction (Sec. 2.3 eq. (sourceeq) bracket, with the Arrhenius
// K_f, K_r = K_f/K_c, third-body [M] and Troe falloff) at temperature T and
// concentrations C: rate_gather then rate_compute.  S is the scalar type
// (double, or Dual for directional derivatives); Vec is any indexable vector of
// S.  NS > 0 fixes the species count at compile time; otherwise Nrt is used.
template <int NS, bool WITH_J, class S, class Vec>
__device__ __forceinline__ void rate_one(const MechView& mv, const double* r, int Nrt, S T, S lnT, S invT,
                                         S lnP0RT, const Vec& C, const Vec& gRT, const Vec& hRT,
                                         RateOutT<S>& o, const SparseEff* se = nullptr) {
  RxIn<S> g;
  rate_gather<NS, WITH_J>(mv, r, Nrt, C, gRT, hRT, g, se);
  rate_compute<NS, WITH_J>(mv, g, T, lnT, invT, lnP0RT, o);
}

// ---------------------------------------------------------------------------
// The fixed-point form of the rates for a mechanism read from its blob (the
// generated kernels have it as literals, gen_fixed in codegen.cu): the exponents
// are 64-bit sums in units of 2^-53 octave, the products of rate constants and
// concentrations unpacked numbers (Fx), so that a reaction's net rate takes the
// FP64 pipe, 64 cycles per warp instruction, only for its collider.
// ---------------------------------------------------------------------------
struct FixState {
  uint64_t L, I, t1, t2, t3, t4;  // log2 T 2^60, 1/T 2^69, T 2^50, T^2 2^36, T^3 2^22, T^4 2^8
  int64_t lp;                     // log2(p_std / (R T)) 2^53
};

__device__ __forceinline__ bool fixed_covers(const MechView& mv, double T) { return T >= mv.T_low && T < FIX_T_HIGH; }

__device__ __forceinline__ FixState fix_state(double T, double invT) {
  FixState s;
  s.L = log2_fixed(T);
  s.I = pos_fixed<69>(invT);
  s.t1 = pos_fixed<50>(T);
  s.t2 = mul_fixed(s.t1, s.t1);
  s.t3 = mul_fixed(s.t2, s.t1);
  s.t4 = mul_fixed(s.t2, s.t2);
  // ln(p_std / R) log2(e) 2^53, from its parts (a literal of the sum)
  s.lp = -(int64_t)0xcb7954cba85db7ll - (int64_t)(s.L >> 7);
  return s;
}

// c times a fixed-point monomial, c signed
__device__ __forceinline__ int64_t fix_term(long long c, uint64_t mono) { return mul_fixed_signed(c, mono); }

// g_k/RT log2(e) 2^53 from the species' record
__device__ __forceinline__ int64_t fix_gibbs(const long long* c, const FixState& s) {
  int64_t v = fix_term(__ldg(c + 2), s.t1) + fix_term(__ldg(c + 3), s.t2) + fix_term(__ldg(c + 6), s.I);
  const long long c3 = __ldg(c + 4), c4 = __ldg(c + 5);
  if (c3 | c4) v += fix_term(c3, s.t3) + fix_term(c4, s.t4);
  return __ldg(c) + fix_term(__ldg(c + 1), s.L) + 4 * v;
}

__device__ __forceinline__ uint32_t hi_word(double x) { return (uint32_t)__double2hiint(x); }

// 2^X as a number, and a number as a factor of fx_mul
__device__ __forceinline__ Fx fx_exp2(int64_t X) {
  Fx a;
  a.m = exp2_parts(X, a.e);
  a.e -= 63;
  return a;
}
__device__ __forceinline__ Fx fx_as_factor(Fx a) {
  a.e += 64;
  return a;
}

// The exponents of reaction j: of k_f (k_inf of a falloff reaction) and of k_r (1 / K_c
// of a falloff reaction; 0 for an irreversible one).  G holds the species' g/RT
// log2(e) 2^53 as 64-bit integers in the doubles' storage.
template <class Vec>
__device__ __forceinline__ void rate_exponents(const MechView& mv, int j, const double* r, const FixState& fs,
                                               const Vec& G, int64_t& x, int64_t& xr) {
  const RxMeta mt = load_meta(r);
  const int nr = mt.nrnp & 15, np = mt.nrnp >> 4;
  const long long* rr = mv.fix + mv.fr + 2 * j;
  x = __ldg(mv.fix + j) + fix_term(__ldg(rr), fs.L) + 4 * fix_term(__ldg(rr + 1), fs.I);
  auto g = [&](int k) { return (int64_t)__double_as_longlong(G[k]); };
  int64_t xc = g(mt.prod[0]) - g(mt.reac[0]) - (np - nr) * fs.lp;
  if (np > 1) xc += g(mt.prod[1]);
  if (np > 2) xc += g(mt.prod[2]);
  if (nr > 1) xc -= g(mt.reac[1]);
  if (nr > 2) xc -= g(mt.reac[2]);
  xr = (mt.flags & 4) == 0 ? 0 : (mt.flags & 3) == 2 ? xc : add_exponents(x, xc);
}

// rate_gather and rate_compute in fixed point: the same results but for rounding.
// se: sparse efficiencies (the warp path), else the dense row.  (The powers of two
// of eight reactions at a time, as in the generated kernels, were slower here: the
// loops wait for the reactions' records; 16411 source terms 76 instead of 64 us.)
template <int NS, bool WITH_J, class Vec>
__device__ __forceinline__ void rate_fixed(const MechView& mv, int j, const double* r, int Nrt, double T, double invT,
                                           const FixState& fs, const Vec& C, const Vec& G, const Vec& hRT, RateOut& o,
                                           const SparseEff* se = nullptr) {
  const int N = NS > 0 ? NS : Nrt;
  int64_t x, xr;
  rate_exponents(mv, j, r, fs, G, x, xr);
  Fx kf = fx_exp2(x), kr = fx_exp2(xr);
  const RxMeta mt = load_meta(r);
  const RxSlots sl = load_slots(r);
  o.active = true;
  o.mt = mt;
  o.sl = sl;
  const int nr = mt.nrnp & 15, np = mt.nrnp >> 4, type = mt.flags & 3;
  const bool rev = (mt.flags & 4) != 0;
  o.cr[0] = C[mt.reac[0]];
  o.cr[1] = nr > 1 ? C[mt.reac[1]] : 1.0;
  o.cr[2] = nr > 2 ? C[mt.reac[2]] : 1.0;
  o.cp[0] = C[mt.prod[0]];
  o.cp[1] = np > 1 ? C[mt.prod[1]] : 1.0;
  o.cp[2] = np > 2 ? C[mt.prod[2]] : 1.0;
  double sh = 0.0;
  if (WITH_J) {
    sh = hRT[mt.prod[0]] - hRT[mt.reac[0]];
    if (np > 1) sh += hRT[mt.prod[1]];
    if (np > 2) sh += hRT[mt.prod[2]];
    if (nr > 1) sh -= hRT[mt.reac[1]];
    if (nr > 2) sh -= hRT[mt.reac[2]];
  }
  double Mc = 1.0;
  if (type != 0) {
    if (se) {
      Mc = se->ctot;
      for (int t = se->off[sl.eff]; t < se->off[sl.eff + 1]; ++t) {
        const int* e = se->ent + 3 * t;
        Mc += __hiloint2double(e[2], e[1]) * C[e[0]];
      }
    } else {
      const double* ef = mv.eff + N * sl.eff;
      Mc = 0.0;
#pragma unroll
      for (int l = 0; l < N; ++l) Mc += ef[l] * C[l];
    }
  }
  const double beta = r[1], EaR = r[2];
  double dlnk = 0.0, gpr = 0.0;
  if (WITH_J) dlnk = fma(EaR, invT, beta) * invT;
  if (type == 2) {
    // Troe falloff, logarithms to base 2 (see rate_compute); kr holds 1 / K_c here
    const double* tr = mv.tr + TR_REC * sl.troe;
    const long long* rt = mv.fix + mv.ff + 3 * sl.troe;
    const int64_t xd = __ldg(rt) + fix_term(__ldg(rt + 1), fs.L) + 4 * fix_term(__ldg(rt + 2), fs.I);
    const double Pr = fx_pack(fx_exp2(xd), 0u) * Mc;
    if (!(Pr >= 0x1p-1022)) {  // no low-pressure rate or no collider: k = 0
      o.active = false;
      return;
    }
    double e3, e1;
    exp_rate2(-T * tr[4], -T * tr[5], e3, e1);
    const double e2 = exp_rate(-tr[6] * invT);
    const double Fc = fma(1.0 - tr[3], e3, fma(tr[3], e1, e2));
    const int64_t lc = log2_q52(Fc);
    // 0.67 2^64, 1.27 2^63, 0.14 2^64
    constexpr uint64_t C067 = 12359318529385400320ull, C127 = 11713682486805565440ull, C014 = 2582544170319337472ull;
    constexpr int64_t Q04 = 5984253652114523ll, Q075 = 11220475597714730ll;  // 0.4 and 0.75 log2(10) 2^52
    const int64_t lx = log2_q52(Pr) - Q04 - mul_fixed_signed(lc, C067), ln = Q075 - 2 * mul_fixed_signed(lc, C127);
    const double xl = q52_to_double(lx), den = q52_to_double(ln - mul_fixed_signed(lx, C014)), Lc = q52_to_double(lc);
    const double den2 = den * den, q1 = den2 * rcp_any(fma(xl, xl, den2)), onePr = rcp_any(1.0 + Pr);
    kf = fx_mul(fx_mul(kf, fx_factor(Pr * onePr)), fx_exp2_factor(Lc * q1));
    kr = fx_mul(kf, fx_as_factor(kr));
    if (WITH_J) {
      const double nn = q52_to_double(ln), rden = rcp_any(den), f1 = xl * rden;
      const double df1_dLc = fma(-0.67, den, -(xl * (-1.27 + 0.67 * 0.14))) * (rden * rden);
      const double g2 = 2.0 * Lc * f1 * q1 * q1;
      gpr = fma(-g2, nn * rden * rden, onePr);  // d ln k / d ln Pr
      const double dFc = fma(-(1.0 - tr[3]) * tr[4], e3, fma(-tr[3] * tr[5], e1, tr[6] * invT * invT * e2));
      const double dlnk0 = fma(tr[2], invT, tr[1]) * invT;
      dlnk = fma(fma(-g2, df1_dLc, q1) * dFc, rcp_any(Fc), fma(gpr, dlnk0 - dlnk, dlnk));
    }
  }
  const uint32_t sf = hi_word(o.cr[0]) ^ hi_word(o.cr[1]) ^ hi_word(o.cr[2]);
  const uint32_t sb = hi_word(o.cp[0]) ^ hi_word(o.cp[1]) ^ hi_word(o.cp[2]);
  const Fx pf = fx_mul(fx_mul(fx_mul(kf, fx_factor(o.cr[0])), fx_factor(o.cr[1])), fx_factor(o.cr[2]));
  Fx pb = fx_mul(fx_mul(fx_mul(kr, fx_factor(o.cp[0])), fx_factor(o.cp[1])), fx_factor(o.cp[2]));
  if (!rev) {
    pb.m = 0;
    pb.e = -100000;  // must not set the scale of the difference
  }
  const double q0 = fx_diff(pf, sf, pb, sb);
  o.q = type == 1 ? Mc * q0 : q0;
  if (WITH_J) {
    const double kfd = fx_pack(kf, 0u), krd = rev ? fx_pack(kr, 0u) : 0.0, pbd = fx_pack(pb, sb);
    o.fk = type == 1 ? Mc * kfd : kfd;
    o.rk = type == 1 ? Mc * krd : krd;
    // dk/d[M] = k gpr / [M] for falloff
    o.dqdM = type == 1 ? q0 : type == 2 ? q0 * (gpr * rcp_any(Mc)) : 0.0;
    const double dlnKc = (sh - (double)(np - nr)) * invT;
    o.dqdT = fma(o.q, dlnk, (type == 1 ? Mc * pbd : pbd) * dlnKc);
  }
}

// Optional accumulation of d/d ln A_j of a weighted sum of the right-hand side
// (the discrete adjoint's parameter gradient), inside eval_vjp.  Mode 1: the
// weights are eval_vjp's cotangent r of dy/dt, i.e. th[j] += r . d f / d ln A_j
// = q_j sum_k nu_kj u_k with u_k = (W_k r_{Y_k} - r_T H_k / cp) / rho.  Mode 2:
// heat release, th[j] += g * d qdot / d ln A_j with qdot = -0.1 sum_k H_k wdot_k
// [W/m^3].  The scratch u may be the storage of eval_vjp's cpR vector: eval_vjp
// reads u only in its reaction loop and writes cpR after it.
struct ThetaHook {
  int mode;        // 0: off
  double g;        // mode 2: weight
  SV th;           // per-thread accumulator, M entries
  SV u;            // per-thread scratch, N entries
};

// Evaluate f = dy/dt for y = (T, Y) and, when WITH_J, the analytic Jacobian
// J = df/dy (row-major in the strided view Jv, n x n with n = NS + 1).
// Constant-pressure reactor (CONSTV false): pc is the pressure [dyn/cm^2], rho
// follows from the ideal-gas law, and the energy balance conserves h.
// Constant-volume reactor (Sec. 2.2, CONSTV true): pc is the fixed density
// [g/cm^3]; U_k = H_k - R T and cv = cp - R/W replace H_k and cp in the
// temperature equation, and C_k = rho Y_k / W_k no longer depends on T or on
// the mean molar mass.  Returns qdot = -sum_k H_k wdot_k (U_k at constant
// volume) in erg/(cm^3 s).
template <int NS, bool WITH_J, class S = double, bool CONSTV = false, int ST = 0>
__device__ __forceinline__ S eval_thread(const MechView& mv, const double pc, const S (&y)[NS + 1], S (&f)[NS + 1],
                                         SVT<S, ST> C, SVT<S, ST> wdot, SVT<S, ST> gRT, SVT<S, ST> hRT,
                                         SVT<S, ST> cpR, SVT<S, ST> Jv) {
  constexpr int n = NS + 1;
  constexpr double EV = CONSTV ? 1.0 : 0.0;  // U/(RT) = H/(RT) - 1, cv/R = cp/R - 1
  const S T = y[0];
  const S invT = 1.0 / T;
  S sumYW(0.0), cpm(0.0);
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    const double* a = mv.sp + SP_REC * k + 2;
    const S cpk = a[0] + T * (a[1] + T * (a[2] + T * (a[3] + T * a[4])));
    cpR[k] = cpk;
    sumYW += y[1 + k] * mv.sp[SP_REC * k + 1];
    cpm += y[1 + k] * (cpk - EV) * mv.sp[SP_REC * k + 1];
  }
  // fixed-point rates where the temperature is covered and the concentrations
  // are finite
  const bool fixed = fixed_covers(mv, T) && rcp_in_range(sumYW) && rcp_in_range(pc);
  FixState fst;
  S lnT(0.0);
  if (fixed) fst = fix_state(T, invT);
  else lnT = fast_log(T);
#pragma unroll 1
  for (int k = 0; k < NS; ++k) {
    const double* a = mv.sp + SP_REC * k + 2;
    const double* ah = mv.sp + SP_REC * k + SP_H;  // a2/2 .. a5/5
    const S hk = a[0] + T * (ah[0] + T * (ah[1] + T * (ah[2] + T * ah[3]))) + a[5] * invT;
    hRT[k] = hk;
    if (fixed) {
      gRT[k] = __longlong_as_double(fix_gibbs(mv.fix + mv.fg + 7 * k, fst));
    } else {
      const double* as = mv.sp + SP_REC * k + SP_S;  // a3/2 .. a5/4
      const S sk = a[0] * lnT + T * (a[1] + T * (as[0] + T * (as[1] + T * as[2]))) + a[6];
      gRT[k] = hk - sk;
    }
  }
  cpm = cpm * RU;  // cp, or cv at constant volume
  const S rho = CONSTV ? S(pc) : pc * invT / (RU * sumYW);
  const S invrho = 1.0 / rho;
  const S invcp = 1.0 / cpm;
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    C[k] = rho * y[1 + k] * mv.sp[SP_REC * k + 1];
    wdot[k] = S(0.0);
  }
  if (WITH_J) {
#pragma unroll
    for (int i = 0; i < n * n; ++i) Jv[i] = S(0.0);
  }
  const S lnP0RT = LOG_PSTD_RU - lnT;
  for (int j = 0; j < mv.M; ++j) {
    RateOutT<S> ro;
    if (fixed) rate_fixed<NS, WITH_J>(mv, j, mv.rx + RX_REC * j, NS, T, invT, fst, C, gRT, hRT, ro);
    else
      rate_one<NS, WITH_J>(mv, mv.rx + RX_REC * j, NS, T, lnT, invT, lnP0RT, C, gRT, hRT, ro);
    if (!ro.active) continue;
    const RxMeta mt = ro.mt;
    const int nr = mt.nrnp & 15, np = mt.nrnp >> 4;
    const S q = ro.q;
    wdot[mt.reac[0]] -= q;
    if (nr > 1) wdot[mt.reac[1]] -= q;
    if (nr > 2) wdot[mt.reac[2]] -= q;
    wdot[mt.prod[0]] += q;
    if (np > 1) wdot[mt.prod[1]] += q;
    if (np > 2) wdot[mt.prod[2]] += q;
    if (WITH_J) {
      // d q / d C of each reactant / product entry (product rule, no division)
      S dr[3], dp[3];
      dr[0] = ro.fk * ro.cr[1] * ro.cr[2];
      dr[1] = ro.fk * ro.cr[0] * ro.cr[2];
      dr[2] = ro.fk * ro.cr[0] * ro.cr[1];
      dp[0] = -(ro.rk * ro.cp[1] * ro.cp[2]);
      dp[1] = -(ro.rk * ro.cp[0] * ro.cp[2]);
      dp[2] = -(ro.rk * ro.cp[0] * ro.cp[1]);
      const int type = mt.flags & 3;
      const double* ef = (type != 0) ? mv.eff + NS * ro.sl.eff : nullptr;
#pragma unroll
      for (int a = 0; a < 6; ++a) {
        const bool isr = a < 3;
        const int ia = isr ? a : a - 3;
        if (ia >= (isr ? nr : np)) continue;
        const double sgn = isr ? -1.0 : 1.0;
        const int row = 1 + (isr ? mt.reac[ia] : mt.prod[ia]);
        Jv[row * n] += sgn * ro.dqdT;
        Jv[row * n + 1 + mt.reac[0]] += sgn * dr[0];
        if (nr > 1) Jv[row * n + 1 + mt.reac[1]] += sgn * dr[1];
        if (nr > 2) Jv[row * n + 1 + mt.reac[2]] += sgn * dr[2];
        Jv[row * n + 1 + mt.prod[0]] += sgn * dp[0];
        if (np > 1) Jv[row * n + 1 + mt.prod[1]] += sgn * dp[1];
        if (np > 2) Jv[row * n + 1 + mt.prod[2]] += sgn * dp[2];
        if (ef) {
          const S cM = sgn * ro.dqdM;
#pragma unroll
          for (int l = 0; l < NS; ++l) Jv[row * n + 1 + l] += cM * ef[l];
        }
      }
    }
  }
  // heat release
  S Hw(0.0);
#pragma unroll
  for (int k = 0; k < NS; ++k) Hw += (hRT[k] - EV) * wdot[k];
  Hw = Hw * (RU * T);
#pragma unroll
  for (int k = 0; k < NS; ++k) f[1 + k] = mv.sp[SP_REC * k] * wdot[k] * invrho;
  f[0] = -(Hw * invrho * invcp);
  if (WITH_J) {
    // species rows: concentration-space Jc[k][l] = d wdot_k / d C_l (stored in
    // Jv[1+k][1+l]) and dwdot_k/dT at fixed C (Jv[1+k][0]) -> (T, Y) space.
    // At constant pressure C also moves with T and with the mean molar mass;
    // at constant volume it does not.
    const S Wbar = 1.0 / sumYW;
#pragma unroll 1
    for (int k = 0; k < NS; ++k) {
      const int row = (1 + k) * n;
      const double Wk = mv.sp[SP_REC * k];
      if (CONSTV) {
#pragma unroll
        for (int i = 0; i < NS; ++i) Jv[row + 1 + i] = Wk * Jv[row + 1 + i] * mv.sp[SP_REC * i + 1];
        Jv[row] = Wk * invrho * Jv[row];
      } else {
        S s(0.0);
#pragma unroll
        for (int l = 0; l < NS; ++l) s += Jv[row + 1 + l] * C[l];
        const S wk = wdot[k];
        const S a = Wk * Wbar * invrho * (wk - s);
#pragma unroll
        for (int i = 0; i < NS; ++i) {
          const double iWi = mv.sp[SP_REC * i + 1];
          Jv[row + 1 + i] = (Wk * Jv[row + 1 + i] + a) * iWi;
        }
        Jv[row] = Wk * invrho * (Jv[row] + (wk - s) * invT);
      }
    }
    // temperature row: f_T = -sum_k e_k f_Yk / c with e_k the specific enthalpy
    // (internal energy) and c = cp (cv)
    S dcp(0.0), cpf(0.0);
#pragma unroll
    for (int k = 0; k < NS; ++k) {
      const double* a = mv.sp + SP_REC * k + 2;
      const double iW = mv.sp[SP_REC * k + 1];
      dcp += y[1 + k] * (a[1] + T * (2.0 * a[2] + T * (3.0 * a[3] + T * 4.0 * a[4]))) * iW;
      cpf += (cpR[k] - EV) * iW * f[1 + k];
    }
    dcp = dcp * RU;
    // (where two products meet in a sum the text says which one is fused: eval_lanes.cuh
    // rounds alike)
#pragma unroll 1
    for (int jc = 0; jc < n; ++jc) {
      S acc(0.0);
#pragma unroll
      for (int k = 0; k < NS; ++k) acc += (hRT[k] - EV) * mv.sp[SP_REC * k + 1] * Jv[(1 + k) * n + jc];
      acc = acc * (RU * T);
      if (jc == 0) {
        Jv[0] = fma(-invcp, fma(cpf, RU, acc), -(f[0] * dcp * invcp));
      } else {
        const double iWj = mv.sp[SP_REC * (jc - 1) + 1];
        const S cpj = RU * (cpR[jc - 1] - EV) * iWj;
        Jv[jc] = fma(-(f[0] * cpj), invcp, -(invcp * acc));
      }
    }
  }
  return -Hw;
}

// b = J(y)^T r for a fixed vector r, without forming J: the transpose of the
// assembly in eval_thread, accumulated reaction by reaction (reverse mode).
// With rho_k = r_{1+k} + r_0 c_k, c_k = -R T h_k/(RT) / (W_k cp) the weight of
// species row k in the temperature row, and sigma_k = W_k rho_k:
//   v_i = sum_k sigma_k dwdot_k/dC_i,   v_T = sum_k sigma_k dwdot_k/dT|_C
// (each reaction adds w_j dq_j/dC_i and w_j dq_j/dT, w_j = sum over its
// products of sigma minus sum over its reactants), D = sum_k sigma_k wdot_k -
// sum_l v_l C_l, and then
//   b_T     = (v_T + D / T) / rho + r_0 e_T
//   b_{Y_i} = (v_i + D Wbar / rho) / W_i + r_0 e_i
// with e the temperature row's own terms (e_T = -(cpf + f_T dcp/dT) / cp,
// e_i = -f_T cp_i / cp).  Also returns f = dy/dt (f may alias nothing) and, with
// a hook, its ln A terms.  sig and v are N-entry scratch vectors; cpR receives
// cp_k/R after the reaction loop (the hook's u may share its storage).
template <int NS>
__device__ __forceinline__ void eval_vjp(const MechView& mv, const double pc, const double (&y)[NS + 1],
                                         const double (&r)[NS + 1], double (&b)[NS + 1], double (&f)[NS + 1], SV C,
                                         SV wdot, SV gRT, SV hRT, SV cpR, SV sig, SV v,
                                         const ThetaHook* hook = nullptr) {
  const double T = y[0];
  const double invT = 1.0 / T;
  double sumYW = 0.0, cpm = 0.0;
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    const double* a = mv.sp + SP_REC * k + 2;
    const double cpk = a[0] + T * (a[1] + T * (a[2] + T * (a[3] + T * a[4])));
    sumYW += y[1 + k] * mv.sp[SP_REC * k + 1];
    cpm += y[1 + k] * cpk * mv.sp[SP_REC * k + 1];
  }
  // the rates in fixed point (rate_fixed) where it covers the state
  FixState fst;
  const bool fixed = fixed_covers(mv, T) && rcp_in_range(sumYW) && rcp_in_range(pc);
  double lnT = 0.0;
  if (fixed) fst = fix_state(T, invT);
  else lnT = fast_log(T);
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    const double* a = mv.sp + SP_REC * k + 2;
    const double* ah = mv.sp + SP_REC * k + SP_H;  // a2/2 .. a5/5
    const double hk = a[0] + T * (ah[0] + T * (ah[1] + T * (ah[2] + T * ah[3]))) + a[5] * invT;
    hRT[k] = hk;
    if (fixed) {
      gRT[k] = __longlong_as_double(fix_gibbs(mv.fix + mv.fg + 7 * k, fst));
    } else {
      const double* as = mv.sp + SP_REC * k + SP_S;  // a3/2 .. a5/4
      const double sk = a[0] * lnT + T * (a[1] + T * (as[0] + T * (as[1] + T * as[2]))) + a[6];
      gRT[k] = hk - sk;
    }
  }
  cpm = cpm * RU;
  const double rho = pc * invT / (RU * sumYW);
  const double invrho = 1.0 / rho;
  const double invcp = 1.0 / cpm;
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    C[k] = rho * y[1 + k] * mv.sp[SP_REC * k + 1];
    wdot[k] = 0.0;
    v[k] = 0.0;
    const double ck = -(invcp * (RU * T) * hRT[k] * mv.sp[SP_REC * k + 1]);
    sig[k] = mv.sp[SP_REC * k] * (r[1 + k] + r[0] * ck);
  }
  // the hook's weights: mode 1, u_k = sigma_k / rho
  if (hook && hook->mode == 2) {
#pragma unroll
    for (int k = 0; k < NS; ++k) hook->u[k] = -0.1 * hook->g * (RU * T * hRT[k]);
  }
  double vT = 0.0;
  const double lnP0RT = LOG_PSTD_RU - lnT;
  for (int j = 0; j < mv.M; ++j) {
    RateOut ro;
    if (fixed) {
      rate_fixed<NS, true>(mv, j, mv.rx + RX_REC * j, NS, T, invT, fst, C, gRT, hRT, ro);
    } else {
      rate_one<NS, true>(mv, mv.rx + RX_REC * j, NS, T, lnT, invT, lnP0RT, C, gRT, hRT, ro);
    }
    if (!ro.active) continue;
    const RxMeta mt = ro.mt;
    const int nr = mt.nrnp & 15, np = mt.nrnp >> 4;
    const double q = ro.q;
    wdot[mt.reac[0]] -= q;
    if (nr > 1) wdot[mt.reac[1]] -= q;
    if (nr > 2) wdot[mt.reac[2]] -= q;
    wdot[mt.prod[0]] += q;
    if (np > 1) wdot[mt.prod[1]] += q;
    if (np > 2) wdot[mt.prod[2]] += q;
    double w = sig[mt.prod[0]] - sig[mt.reac[0]];
    if (np > 1) w += sig[mt.prod[1]];
    if (np > 2) w += sig[mt.prod[2]];
    if (nr > 1) w -= sig[mt.reac[1]];
    if (nr > 2) w -= sig[mt.reac[2]];
    if (hook && hook->mode == 1) hook->th[j] += q * (w * invrho);
    if (hook && hook->mode == 2) {
      double wu = hook->u[mt.prod[0]] - hook->u[mt.reac[0]];
      if (np > 1) wu += hook->u[mt.prod[1]];
      if (np > 2) wu += hook->u[mt.prod[2]];
      if (nr > 1) wu -= hook->u[mt.reac[1]];
      if (nr > 2) wu -= hook->u[mt.reac[2]];
      hook->th[j] += q * wu;
    }
    vT += w * ro.dqdT;
    const double wf = w * ro.fk, wr = -(w * ro.rk);
    auto add = [&](int m, const uint8_t* id, double x, const double* c) {
      if (m == 1) {
        v[id[0]] += x;
      } else if (m == 2) {
        v[id[0]] += x * c[1];
        v[id[1]] += x * c[0];
      } else {
        v[id[0]] += x * (c[1] * c[2]);
        v[id[1]] += x * (c[0] * c[2]);
        v[id[2]] += x * (c[0] * c[1]);
      }
    };
    add(nr, mt.reac, wf, ro.cr);
    add(np, mt.prod, wr, ro.cp);
    const int type = mt.flags & 3;
    if (type != 0) {
      const double* ef = mv.eff + NS * ro.sl.eff;
      const double wM = w * ro.dqdM;
#pragma unroll
      for (int l = 0; l < NS; ++l) v[l] += wM * ef[l];
    }
  }
  // cp_k/R, recomputed (the same arithmetic as in the first loop) now that the
  // hook's scratch is no longer read
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    const double* a = mv.sp + SP_REC * k + 2;
    cpR[k] = a[0] + T * (a[1] + T * (a[2] + T * (a[3] + T * a[4])));
  }
  double Hw = 0.0, sw = 0.0, svc = 0.0;
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    Hw += hRT[k] * wdot[k];
    sw += sig[k] * wdot[k];
    svc += v[k] * C[k];
  }
  Hw = Hw * (RU * T);
#pragma unroll
  for (int k = 0; k < NS; ++k) f[1 + k] = mv.sp[SP_REC * k] * wdot[k] * invrho;
  f[0] = -(Hw * invrho * invcp);
  double dcp = 0.0, cpf = 0.0;
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    const double* a = mv.sp + SP_REC * k + 2;
    const double iW = mv.sp[SP_REC * k + 1];
    dcp += y[1 + k] * (a[1] + T * (2.0 * a[2] + T * (3.0 * a[3] + T * 4.0 * a[4]))) * iW;
    cpf += cpR[k] * iW * f[1 + k];
  }
  dcp = dcp * RU;
  cpf = cpf * RU;
  const double D = sw - svc;
  const double Wbar = 1.0 / sumYW;
  b[0] = invrho * (vT + invT * D) - r[0] * (invcp * (cpf + f[0] * dcp));
  const double DW = Wbar * invrho * D;
  const double fcp = r[0] * f[0] * invcp * RU;
#pragma unroll
  for (int i = 0; i < NS; ++i) {
    const double iWi = mv.sp[SP_REC * i + 1];
    b[1 + i] = (v[i] + DW) * iWi - fcp * cpR[i] * iWi;
  }
}

// The second-derivative terms of the reverse sweep over one Rosenbrock step:
//   b += grad_y G,  th_j += dG/d ln A_j,  G(y) = sum_s r_s . J(y) K_s
// (J = df/dy, r_s the stages' cotangents): d/de [J(y + e K_s)^T r_s] summed over
// the stages, since both are the second derivatives of f contracted with r_s and
// K_s.  All stages act on J at the same y, so one pass over the reactions does:
//   r_s . f = sum_k u_k wdot_k,  u_k = (W_k r_k - r_T H_k / cp) / rho,
//   G = sum_j [q_T z_T + sum_l q_{C_l} z_l] - sum_k omega_k wdot_k
//       - (A1 Hc / cp + f_T rho A2 / cp) / rho
// with z_j = sum_k nu_kj Z_k, Z_k = sum_s u_k (K_T, dC_1 .. dC_N), dC the change of
// the concentrations along K (dC_l = rho K_l / W_l + C_l theta, theta = -(K_T/T +
// S_K/S), S = sum Y_l/W_l), omega_k = sum_s u_k theta, A1 = sum_s r_T K_T,
// A2 = sum_s r_T dcp, Hc = sum_k wdot_k Cp_k.  Per reaction: q and its first
// derivatives as Duals along z_j, whose derivative halves are the gradient of
// q_T z_T + sum q_C z_C.  A Dual evaluation per stage (six per step, each with
// every exponential and every species sum in Duals) took two thirds of the sweep:
// gradients of 65536 cells, 25 reactions, with the integration 9.57 -> 6.44 ms (6.07 with the ordered sum of the
// ln A partials in parallel and eval_vjp's weights shared).
// K: element i of stage s at K[s n + i]; R likewise.  v, wdot, ...: scratch of NS.
template <int NS, class KView>
__device__ __forceinline__ void second_order(const MechView& mv, const double pc, const double (&y)[NS + 1], int ns,
                                             const KView& K, const SV& R, double (&b)[NS + 1], SV C, SV wdot, SV gRT,
                                             SV hRT, SV cpR, SV v, SV th) {
  constexpr int n = NS + 1, ZC = n + 1;  // a row of Z: z_T, z_1 .. z_N, omega
  const double T = y[0], invT = 1.0 / T, lnT = fast_log(T), lnP0RT = LOG_PSTD_RU - lnT;
  double S = 0.0, cp = 0.0, dcp = 0.0;
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    const double* a = mv.sp + SP_REC * k + 2;
    const double* ah = mv.sp + SP_REC * k + SP_H;
    const double* as = mv.sp + SP_REC * k + SP_S;
    const double iW = mv.sp[SP_REC * k + 1];
    const double cpk = a[0] + T * (a[1] + T * (a[2] + T * (a[3] + T * a[4])));
    const double hk = a[0] + T * (ah[0] + T * (ah[1] + T * (ah[2] + T * ah[3]))) + a[5] * invT;
    const double sk = a[0] * lnT + T * (a[1] + T * (as[0] + T * (as[1] + T * as[2]))) + a[6];
    cpR[k] = cpk;
    hRT[k] = hk;
    gRT[k] = hk - sk;
    S += y[1 + k] * iW;
    cp += y[1 + k] * cpk * iW;
    dcp += y[1 + k] * (a[1] + T * (2.0 * a[2] + T * (3.0 * a[3] + T * 4.0 * a[4]))) * iW;
  }
  cp *= RU;
  dcp *= RU;
  const double invS = 1.0 / S, rho = pc * invT / (RU * S), vol = 1.0 / rho, icp = 1.0 / cp, RT = RU * T;
  double Z[NS * ZC], t[NS];
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    C[k] = rho * y[1 + k] * mv.sp[SP_REC * k + 1];
    wdot[k] = 0.0;
    v[k] = 0.0;
    t[k] = 0.0;
  }
#pragma unroll 1
  for (int i = 0; i < NS * ZC; ++i) Z[i] = 0.0;
  double A1 = 0.0, A2 = 0.0, A3 = 0.0;
#pragma unroll 1
  for (int s = 0; s < ns; ++s) {
    const double KT = K[s * n], rT = R[s * n];
    double X[NS], SK = 0.0, dc = 0.0;
#pragma unroll
    for (int l = 0; l < NS; ++l) {
      X[l] = K[s * n + 1 + l] * mv.sp[SP_REC * l + 1];
      SK += X[l];
      dc += X[l] * cpR[l];
    }
    const double theta = -(KT * invT + SK * invS);
    A1 += rT * KT;
    A2 += rT * (RU * dc + KT * dcp);
    A3 += rT * theta;
#pragma unroll
    for (int l = 0; l < NS; ++l) {
      X[l] = rho * X[l] + C[l] * theta;
      t[l] += rT * X[l];
    }
    const double rH = rT * RT * icp;
#pragma unroll 1
    for (int k = 0; k < NS; ++k) {
      const double u = vol * (mv.sp[SP_REC * k] * R[s * n + 1 + k] - rH * hRT[k]);
      double* z = Z + k * ZC;
      z[0] += u * KT;
#pragma unroll
      for (int l = 0; l < NS; ++l) z[1 + l] += u * X[l];
      z[n] += u * theta;
    }
  }
  // weights of q_j's own derivatives from the terms with wdot: sum nu (cA cpR + cB hRT) - omega_j
  const double cA = -vol * icp * A1 * RU, cB = vol * icp * icp * A2 * RT;
  double G1T = 0.0, kw = 0.0, kT = 0.0, Q1 = 0.0, Q2 = 0.0, gT = 0.0;
#pragma unroll 1
  for (int j = 0; j < mv.M; ++j) {
    const double* rx = mv.rx + RX_REC * j;
    RxIn<double> g;
    rate_gather<NS, true>(mv, rx, NS, C, gRT, hRT, g);
    if (g.lnA == -INFINITY) continue;
    const RxMeta mt = g.mt;
    const int nr = mt.nrnp & 15, np = mt.nrnp >> 4, type = mt.flags & 3, dnu = np - nr;
    auto col = [&](int m) {
      double z = Z[mt.prod[0] * ZC + m] - Z[mt.reac[0] * ZC + m];
      if (np > 1) z += Z[mt.prod[1] * ZC + m];
      if (np > 2) z += Z[mt.prod[2] * ZC + m];
      if (nr > 1) z -= Z[mt.reac[1] * ZC + m];
      if (nr > 2) z -= Z[mt.reac[2] * ZC + m];
      return z;
    };
    double scp = cpR[mt.prod[0]] - cpR[mt.reac[0]];
    if (np > 1) scp += cpR[mt.prod[1]];
    if (np > 2) scp += cpR[mt.prod[2]];
    if (nr > 1) scp -= cpR[mt.reac[1]];
    if (nr > 2) scp -= cpR[mt.reac[2]];
    const double zT = col(0), om = col(n), gw = cA * scp + cB * g.sh;
    Dual Mc(1.0), cr[3], cpd[3];
    double Mt = 0.0;
    const double* ef = nullptr;
    if (type != 0) {
      ef = mv.eff + NS * load_slots(rx).eff;
      Mc = Dual(g.Mc);
#pragma unroll 1
      for (int l = 0; l < NS; ++l) {
        Mc.d += ef[l] * col(1 + l);
        Mt += ef[l] * t[l];
      }
    }
    cr[0] = Dual(g.cr[0], col(1 + mt.reac[0]));
    cpd[0] = Dual(g.cp[0], col(1 + mt.prod[0]));
    cr[1] = cr[2] = cpd[1] = cpd[2] = Dual(1.0);
    if (nr > 1) cr[1] = Dual(g.cr[1], col(1 + mt.reac[1]));
    if (nr > 2) cr[2] = Dual(g.cr[2], col(1 + mt.reac[2]));
    if (np > 1) cpd[1] = Dual(g.cp[1], col(1 + mt.prod[1]));
    if (np > 2) cpd[2] = Dual(g.cp[2], col(1 + mt.prod[2]));
    Dual fk, rk, qT, qM(0.0), q;
    double dl = 0.0, dlr = 0.0, ddl = 0.0, ddlr = 0.0;
    if (type == 2) {
      RxIn<Dual> gd;
      gd.lnA = g.lnA;
      gd.beta = g.beta;
      gd.EaR = g.EaR;
      gd.mt = mt;
      gd.sl = g.sl;
      for (int i = 0; i < 3; ++i) {
        gd.cr[i] = cr[i];
        gd.cp[i] = cpd[i];
      }
      gd.sg = Dual(g.sg, -g.sh * invT * zT);
      gd.sh = Dual(g.sh, (scp - g.sh) * invT * zT);
      gd.Mc = Mc;
      RateOutT<Dual> ro;
      rate_compute<NS, true>(mv, gd, Dual(T, zT), Dual(lnT, zT * invT), Dual(invT, -zT * invT * invT),
                             Dual(lnP0RT, -zT * invT), ro);
      if (!ro.active) continue;
      fk = ro.fk;
      rk = ro.rk;
      qT = ro.dqdT;
      qM = ro.dqdM;
    } else {
      const double lnkf = g.lnA + g.beta * lnT - g.EaR * invT;
      double kf, kr;
      exp_pair(lnkf, lnkf + (dnu == 0 ? g.sg : g.sg - (double)dnu * lnP0RT), kf, kr);
      if ((mt.flags & 4) == 0) kr = 0.0;
      // d ln k / dT of both directions and their derivatives
      const double e = g.EaR * invT, i2 = invT * invT;
      dl = (g.beta + e) * invT;
      ddl = -(g.beta + 2.0 * e) * i2;
      dlr = dl - (g.sh - (double)dnu) * invT;
      ddlr = ddl - (scp - 2.0 * g.sh + (double)dnu) * i2;
      fk = Dual(kf, kf * (dl * zT));
      rk = Dual(kr, kr * (dlr * zT));
    }
    // the derivatives by the concentrations, and both directions' rates
    Dual xr[3], xp[3];
    auto side = [](int m, const Dual& k, const Dual (&c)[3], Dual (&x)[3]) {
      if (m == 1) {
        x[0] = k;
      } else if (m == 2) {
        x[0] = k * c[1];
        x[1] = k * c[0];
      } else {
        x[0] = k * (c[1] * c[2]);
        x[1] = k * (c[0] * c[2]);
        x[2] = k * (c[0] * c[1]);
      }
      return x[0] * c[0];
    };
    Dual F = side(nr, fk, cr, xr), B = side(np, rk, cpd, xp);
    if (type == 1) {
      qM = F - B;
      F *= Mc;
      B *= Mc;
      for (int i = 0; i < 3; ++i) {
        if (i < nr) xr[i] *= Mc;
        if (i < np) xp[i] *= Mc;
      }
    }
    q = F - B;
    if (type != 2) qT = Dual(dl * F.v - dlr * B.v, dl * F.d - dlr * B.d + zT * (ddl * F.v - ddlr * B.v));
    double e = A1 * qT.v + Mt * qM.v, d = (double)nr * F.v - (double)np * B.v + qM.v * Mc.v;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      if (i < nr) {
        v[mt.reac[i]] += xr[i].d + gw * xr[i].v;
        wdot[mt.reac[i]] -= q.v;
        e += t[mt.reac[i]] * xr[i].v;
      }
      if (i < np) {
        v[mt.prod[i]] -= xp[i].d + gw * xp[i].v;
        wdot[mt.prod[i]] += q.v;
        e -= t[mt.prod[i]] * xp[i].v;
      }
    }
    if (type != 0) {
      const double m = qM.d + gw * qM.v;
#pragma unroll
      for (int l = 0; l < NS; ++l) v[l] += m * ef[l];
    }
    gT += qT.d + qT.v * (gw - om);
    th[j] += q.d + q.v * (gw - om);
    G1T += qT.v * zT;
    kw += om * d;
    kT += zT * d;
    Q1 += g.sh * e;
    Q2 += scp * e;
  }
  Q1 *= RT;
  Q2 *= RU;
  double Hw = 0.0, Hc = 0.0, Hcc = 0.0, Ww = 0.0, WZ = 0.0, D = 0.0, dA2 = 0.0;
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    const double* a = mv.sp + SP_REC * k + 2;
    const double iW = mv.sp[SP_REC * k + 1], w = wdot[k];
    const double c1 = a[1] + T * (2.0 * a[2] + T * (3.0 * a[3] + T * 4.0 * a[4]));
    const double c2 = 2.0 * a[2] + T * (6.0 * a[3] + T * 12.0 * a[4]);
    Hw += hRT[k] * w;
    Hc += cpR[k] * w;
    Hcc += c1 * w;
    Ww += Z[k * ZC + n] * w;
    WZ += Z[k * ZC] * w;
    D += v[k] * C[k];
    dA2 += (t[k] - C[k] * A3) * vol * c1 + A1 * y[1 + k] * c2 * iW;
  }
  Hw *= RT;
  Hc *= RU;
  Hcc *= RU;
  dA2 *= RU;
  const double vi = vol * icp, vii = vi * icp;
  const double Gb = -vi * A1 * Hc, Gc = vii * A2 * Hw;
  const double Pv = G1T + kw - Ww + Gb + Gc - D;  // times d ln vol
  const double Pc = vii * (Q1 - A3 * Hw) - icp * (Gb + 2.0 * Gc);
  const double th1 = invT * (kT - WZ);
  b[0] += Pv * invT + Pc * dcp + invT * th1 + gT + vi * (A3 * Hc - Q2 - A1 * Hcc) + vii * (A2 * Hc + Hw * dA2);
  const double Py = (Pv - (kw - Ww) - th1) * invS, H1 = vii * Hw * A1;
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    const double* a = mv.sp + SP_REC * k + 2;
    const double c1 = a[1] + T * (2.0 * a[2] + T * (3.0 * a[3] + T * 4.0 * a[4]));
    b[1 + k] += mv.sp[SP_REC * k + 1] * (Py + rho * v[k] + RU * (Pc * cpR[k] + H1 * c1));
  }
}

// LU with partial pivoting of the n x n matrix in the strided view A; whole rows
// are swapped, the reciprocal of each pivot replaces the diagonal.  The matrix
// stays in shared memory, so the pivot loop is not unrolled (register budget).
template <int n, int ST = 0>
__device__ __forceinline__ bool lu_factor(SVT<double, ST> A, int* piv) {
  bool ok = true;
#pragma unroll 1
  for (int k = 0; k < n; ++k) {
    // pivot search on the magnitudes' bit patterns as 64-bit integers
    // (non-negative doubles order like their patterns): integer compares
    // instead of FP64 ones on the narrow pipe; a NaN sorts above every finite
    // value, is picked, and fails the finiteness test
    int p = k;
    long long best = __double_as_longlong(A[k * n + k]) & 0x7FFFFFFFFFFFFFFFLL;
    for (int i = k + 1; i < n; ++i) {
      const long long v = __double_as_longlong(A[i * n + k]) & 0x7FFFFFFFFFFFFFFFLL;
      if (v > best) { best = v; p = i; }
    }
    piv[k] = p;
    ok = ok && (best > 0) && (best < 0x7FF0000000000000LL);
    if (p != k) {
#pragma unroll
      for (int j = 0; j < n; ++j) {
        const double t = A[k * n + j];
        A[k * n + j] = A[p * n + j];
        A[p * n + j] = t;
      }
    }
    const double inv = rcp_any(A[k * n + k]);
    A[k * n + k] = inv;
    for (int i = k + 1; i < n; ++i) {
      const double l = A[i * n + k] * inv;
      A[i * n + k] = l;
#pragma unroll 4
      for (int j = k + 1; j < n; ++j) A[i * n + j] -= l * A[k * n + j];
    }
  }
  return ok;
}

// Solve in place on the strided vector x with the factors of lu_factor: the
// whole row permutation first, then the unit-lower and upper solves.
template <int n, int ST = 0>
__device__ __forceinline__ void lu_solve(SVT<double, ST> A, const int* piv, SVT<double, ST> x) {
#pragma unroll
  for (int k = 0; k < n; ++k) {
    const int p = piv[k];
    if (p != k) {
      const double t = x[k];
      x[k] = x[p];
      x[p] = t;
    }
  }
#pragma unroll
  for (int k = 0; k < n; ++k) {
    const double xk = x[k];
#pragma unroll
    for (int i = k + 1; i < n; ++i) x[i] -= A[i * n + k] * xk;
  }
#pragma unroll
  for (int k = n - 1; k >= 0; --k) {
    double acc = x[k];
#pragma unroll
    for (int j = k + 1; j < n; ++j) acc -= A[k * n + j] * x[j];
    x[k] = acc * A[k * n + k];
  }
}

}  // namespace df
