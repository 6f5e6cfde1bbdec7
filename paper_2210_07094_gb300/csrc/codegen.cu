// Mechanism-specific thread-per-cell integrator, generated and compiled at run
// time.
//
// The mechanism-independent kernel reads each reaction's species indices,
// stoichiometry and type from the mechanism blob and keeps the per-thread
// species vectors (C, wdot, g/RT, h/RT, cp/R) in shared memory, because those
// indices are only known at run time.  For a loaded mechanism the library can
// instead emit the evaluation of f and J as straight-line code with the
// species indices, the reactant / product counts, the reaction types and the
// mechanism's numbers as literals (ln A is still read from the blob, so
// df_mech_set_lnA keeps working), compile it with NVRTC into a module holding
// the same persistent kernel (integrate_thread.cuh) with that evaluation
// policy, and launch it through the driver API.  The species vectors then live
// in registers, no reaction metadata is decoded and no branch depends on the
// reaction, and the shared memory per thread drops to W and one vector.
//
// Two evaluations are generated.  gen_fixed forms the exponents of the rate
// constants in fixed point and is what cells run; gen_eval, the
// mechanism-independent operations in FP64, takes the states outside the
// fixed-point range (temperatures, ln A, states that are not finite).  Both
// agree with the mechanism-independent kernel to rounding.
//
// NVRTC is opened at run time (dlopen); the driver entry points come through
// cudaGetDriverEntryPointByVersion.  If either is missing, the headers cannot
// be found, or the compilation fails, the integrator uses the
// mechanism-independent kernel and df_chem_jit_info reports why.
#include <dlfcn.h>
#include <sys/stat.h>
#include <unistd.h>

#include <cuda.h>

#include <algorithm>
#include <chrono>
#include <cstdio>
#include <map>
#include <mutex>
#include <sstream>
#include <string>
#include <vector>

#include "common.cuh"
#include "integrate_thread.cuh"
#include "reactions.cuh"

namespace df {

namespace {

// ---------------------------------------------------------------------------
// source generation
// ---------------------------------------------------------------------------
// exact decimal-free spelling of a double (C++17 hexadecimal literal)
std::string lit(double v) {
  if (v == -INFINITY) return "(-INFINITY)";  // ln A0 - ln A of a falloff reaction without a rate
  char b[64];
  snprintf(b, sizeof b, "%a", v);
  return std::string("(") + b + ")";
}

// Horner form c[0] + x (c[1] + x (c[2] + ...)) with the trailing coefficients
// that are exactly zero dropped (for finite x they add exactly zero)
std::string horner(const std::vector<double>& c, const char* x) {
  int top = (int)c.size() - 1;
  while (top > 0 && c[top] == 0.0) --top;
  std::string e = lit(c[top]);
  for (int i = top - 1; i >= 0; --i) e = lit(c[i]) + " + " + x + " * (" + e + ")";
  return e;
}

// f and J of the loaded mechanism as straight-line code: the mechanism-
// independent eval_thread (chem_thread.cuh) at constant pressure with every
// reaction's indices and type resolved and the mechanism's numbers as literals
// (except ln A, read from the blob so that df_mech_set_lnA applies), in the
// same order of operations
void emit_eval(std::ostringstream& o, const df_mech* m) {
  const int N = m->dims.N, n = N + 1, M = m->dims.M;
  o << "template <bool WITH_J, int ST>\n"
    << "__device__ __forceinline__ double gen_eval(const MechView& mv, const double pc, const double (&y)[" << n
    << "], double (&f)[" << n << "], SVT<double, ST> Jv, SVT<double, ST> sM) {\n"
    << "  constexpr int NS = " << N << ";\n  constexpr int n = NS + 1;\n"
    << "  const double T = y[0];\n  const double lnT = fast_log(T);\n  const double invT = 1.0 / T;\n"
    << "  double C[NS], wdot[NS], gRT[NS], hRT[NS], cpW[NS];  // cpW: cp_k / (R W_k)\n"
    << "  double sumYW = 0.0, cpm = 0.0;\n";
  auto sp = [&](int k, int i) { return m->blob_host[m->dims.off_sp + SP_REC * k + i]; };
  for (int k = 0; k < N; ++k) {
    const std::vector<double> a = {sp(k, 2), sp(k, 3), sp(k, 4), sp(k, 5), sp(k, 6)};
    // cp_k / (R W_k) directly: the NASA-7 coefficients times 1 / W_k
    std::vector<double> aw(a);
    for (double& v : aw) v *= sp(k, 1);
    const std::vector<double> ah = {sp(k, SP_H), sp(k, SP_H + 1), sp(k, SP_H + 2), sp(k, SP_H + 3)};
    const std::vector<double> as = {sp(k, SP_S), sp(k, SP_S + 1), sp(k, SP_S + 2)};
    std::vector<double> hs = {sp(k, 2)};
    hs.insert(hs.end(), ah.begin(), ah.end());
    // g/RT = h/RT - s/R in one polynomial: (a1 - a7) - a1 ln T
    // + T (-a2/2 + T (-a3/6 + T (-a4/12 + T (-a5/20)))) + a6 / T
    const std::vector<double> gs = {-0.5 * a[1], -a[2] / 6.0, -a[3] / 12.0, -a[4] / 20.0};
    o << "  {  // species " << k << "\n"
      << "    const double cpw = " << horner(aw, "T") << ";\n    cpW[" << k << "] = cpw;\n"
      << "    const double hk = " << horner(hs, "T") << " + " << lit(sp(k, 7)) << " * invT;\n"
      << "    const double gk = " << lit(sp(k, 2) - sp(k, 8)) << " + " << lit(-sp(k, 2)) << " * lnT + T * ("
      << horner(gs, "T") << ") + " << lit(sp(k, 7)) << " * invT;\n"
      << "    hRT[" << k << "] = hk;\n    gRT[" << k << "] = gk;\n"
      << "    sumYW += y[" << 1 + k << "] * " << lit(sp(k, 1)) << ";\n"
      << "    cpm += y[" << 1 + k << "] * cpw;\n  }\n";
  }
  o << "  cpm = cpm * RU;\n"
    << "  const double rho = pc * invT / (RU * sumYW);\n"
    << "  const double invrho = 1.0 / rho;\n  const double invcp = 1.0 / cpm;\n";
  for (int k = 0; k < N; ++k)
    o << "  C[" << k << "] = rho * y[" << 1 + k << "] * " << lit(sp(k, 1)) << ";\n  wdot[" << k << "] = 0.0;\n";
  // [M] = sum_l eps_l C_l of the third-body and falloff reactions as the sum of
  // all concentrations (once) plus (eps_l - 1) C_l where eps_l is not 1 (exact
  // literals: eps_l - 1 rounds to nothing for eps_l >= 1/2)
  bool any_collider = false;
  for (int j = 0; j < M; ++j) any_collider = any_collider || (meta_of(m, j).flags & 3) != 0;
  if (any_collider) {
    o << "  double ctot = C[0];\n";
    for (int k = 1; k < N; ++k) o << "  ctot += C[" << k << "];\n";
  }
  o
    << "  if (WITH_J) {\n#pragma unroll\n    for (int i = 0; i < n * n; ++i) Jv[i] = 0.0;\n";
  // the unit part of the collider efficiencies, sum over reactions of
  // nu_k d q / d[M], one value per row (sM, the stage vectors' storage, idle
  // while J is built); the conversion below adds it to every column
  if (any_collider) o << "#pragma unroll\n    for (int k = 0; k < NS; ++k) sM[k] = 0.0;\n";
  o << "  }\n"
    << "  const double lnP0RT = LOG_PSTD_RU - lnT;\n";
  for (int j = 0; j < M; ++j) {
    const RxMeta mt = meta_of(m, j);
    const RxSlots sl = slots_of(m, j);
    const int nr = mt.nrnp & 15, np = mt.nrnp >> 4, type = mt.flags & 3;
    const int r[3] = {mt.reac[0], mt.reac[1], mt.reac[2]};
    const int p[3] = {mt.prod[0], mt.prod[1], mt.prod[2]};
    o << "  {  // reaction " << j << "\n"
      << "    RxIn<double> g;\n    const double* r = mv.rx + RX_REC * " << j << ";\n"
      << "    g.lnA = r[0];\n    g.beta = " << lit(m->blob_host[m->dims.off_rx + RX_REC * j + 1])
      << ";\n    g.EaR = " << lit(m->blob_host[m->dims.off_rx + RX_REC * j + 2]) << ";\n";
    for (int i = 0; i < 3; ++i) o << "    g.mt.reac[" << i << "] = " << r[i] << ";\n";
    for (int i = 0; i < 3; ++i) o << "    g.mt.prod[" << i << "] = " << p[i] << ";\n";
    o << "    g.mt.nrnp = " << (int)mt.nrnp << ";\n    g.mt.flags = " << (int)mt.flags << ";\n"
      << "    g.sl.eff = " << sl.eff << ";\n    g.sl.troe = " << sl.troe << ";\n";
    for (int i = 0; i < 3; ++i)
      o << "    g.cr[" << i << "] = " << (i < nr ? "C[" + std::to_string(r[i]) + "]" : std::string("1.0")) << ";\n";
    for (int i = 0; i < 3; ++i)
      o << "    g.cp[" << i << "] = " << (i < np ? "C[" + std::to_string(p[i]) + "]" : std::string("1.0")) << ";\n";
    // sum nu g/RT and h/RT in rate_gather's order
    o << "    double sg = gRT[" << p[0] << "] - gRT[" << r[0] << "];\n"
      << "    double sh = 0.0;\n    if (WITH_J) sh = hRT[" << p[0] << "] - hRT[" << r[0] << "];\n";
    for (int i = 1; i < np; ++i) o << "    sg += gRT[" << p[i] << "];\n    if (WITH_J) sh += hRT[" << p[i] << "];\n";
    for (int i = 1; i < nr; ++i) o << "    sg -= gRT[" << r[i] << "];\n    if (WITH_J) sh -= hRT[" << r[i] << "];\n";
    o << "    g.sg = sg;\n    g.sh = sh;\n";
    auto eff = [&](int l) { return m->blob_host[m->dims.off_eff + N * sl.eff + l]; };
    if (type != 0) {
      o << "    {\n      double Mc = ctot;\n";
      for (int l = 0; l < N; ++l)
        if (eff(l) != 1.0) o << "      Mc += " << lit(eff(l) - 1.0) << " * C[" << l << "];\n";
      o << "      g.Mc = Mc;\n    }\n";
    } else {
      o << "    g.Mc = 0.0;\n";
    }
    if (type == 2) {  // the falloff parameters as literals too (a one-record table)
      const double* tr = &m->blob_host[m->dims.off_tr + TR_REC * sl.troe];
      o << "    const double trp[" << TR_REC << "] = {";
      for (int i = 0; i < TR_REC; ++i) o << (i ? ", " : "") << lit(tr[i]);
      o << "};\n    MechView mvt = mv;\n    mvt.tr = trp;\n    g.sl.troe = 0;\n"
        << "    RateOutT<double> ro;\n    rate_compute<NS, WITH_J>(mvt, g, T, lnT, invT, lnP0RT, ro);\n";
    } else {
      o << "    RateOutT<double> ro;\n    rate_compute<NS, WITH_J>(mv, g, T, lnT, invT, lnP0RT, ro);\n";
    }
    // The species of the reaction with their net stoichiometric coefficient
    // nu_k (products minus reactants): one update of wdot and of each Jacobian
    // row per species, scaled by nu_k, instead of one per reactant or product
    // entry (a species entered twice, or on both sides, is touched once or not
    // at all).  The columns d q / d C_l likewise sum the entries of species l.
    std::vector<int> spc;
    std::vector<int> nu(N, 0);
    for (int i = 0; i < nr; ++i) nu[r[i]] -= 1;
    for (int i = 0; i < np; ++i) nu[p[i]] += 1;
    for (int i = 0; i < nr; ++i)
      if (std::find(spc.begin(), spc.end(), r[i]) == spc.end()) spc.push_back(r[i]);
    for (int i = 0; i < np; ++i)
      if (std::find(spc.begin(), spc.end(), p[i]) == spc.end()) spc.push_back(p[i]);
    auto nu_times = [](int v, const std::string& x) {
      return v == 1 ? "(" + x + ")" : v == -1 ? "-(" + x + ")" : std::to_string(v) + ".0 * (" + x + ")";
    };
    o << "    if (ro.active) {\n      const double q = ro.q;\n";
    for (int k : spc)
      if (nu[k] != 0) o << "      wdot[" << k << "] += " << nu_times(nu[k], "q") << ";\n";
    o << "      if (WITH_J) {\n"
      << "        const double dr0 = ro.fk * ro.cr[1] * ro.cr[2];\n"
      << "        const double dr1 = ro.fk * ro.cr[0] * ro.cr[2];\n"
      << "        const double dr2 = ro.fk * ro.cr[0] * ro.cr[1];\n"
      << "        const double dp0 = -(ro.rk * ro.cp[1] * ro.cp[2]);\n"
      << "        const double dp1 = -(ro.rk * ro.cp[0] * ro.cp[2]);\n"
      << "        const double dp2 = -(ro.rk * ro.cp[0] * ro.cp[1]);\n"
      << "        (void)dr1; (void)dr2; (void)dp1; (void)dp2;\n";
    // d q / d C_l of each species of the reaction
    for (int l : spc) {
      std::string terms;
      for (int i = 0; i < nr; ++i)
        if (r[i] == l) terms += (terms.empty() ? "" : " + ") + std::string("dr") + std::to_string(i);
      for (int i = 0; i < np; ++i)
        if (p[i] == l) terms += (terms.empty() ? "" : " + ") + std::string("dp") + std::to_string(i);
      o << "        const double dq" << l << " = " << terms << ";\n";
    }
    // the concentration-space entries d wdot_k / d C_l enter row k scaled by
    // W_k / W_l (a literal), the column scaling of the conversion to mass
    // fractions below, so that the conversion adds only its rank-one part
    auto wk_over_wl = [&](int k, int l) { return sp(k, 0) * sp(l, 1); };  // W_k * (1 / W_l)
    for (int k : spc) {
      if (nu[k] == 0) continue;
      const int row = 1 + k;
      o << "        Jv[" << row * n << "] += " << nu_times(nu[k], "ro.dqdT") << ";\n";
      for (int l : spc) {
        if (l == k)
          o << "        Jv[" << row * n + 1 + l << "] += " << nu_times(nu[k], "dq" + std::to_string(l)) << ";\n";
        else
          o << "        Jv[" << row * n + 1 + l << "] += " << lit(nu[k] * wk_over_wl(k, l)) << " * dq" << l << ";\n";
      }
      if (type != 0) {
        o << "        {\n          const double cM = " << nu_times(nu[k], "ro.dqdM") << ";\n"
          << "          sM[" << k << "] += cM;\n";
        for (int l = 0; l < N; ++l) {
          if (eff(l) == 1.0) continue;
          const double c = l == k ? eff(l) - 1.0 : (eff(l) - 1.0) * wk_over_wl(k, l);
          o << "          Jv[" << row * n + 1 + l << "] += cM * " << lit(c) << ";\n";
        }
        o << "        }\n";
      }
    }
    o << "      }\n    }\n  }\n";
  }
  o << "  double Hw = 0.0;\n#pragma unroll\n  for (int k = 0; k < NS; ++k) Hw += hRT[k] * wdot[k];\n"
    << "  Hw = Hw * (RU * T);\n"
    ;
  for (int k = 0; k < N; ++k) o << "  f[" << 1 + k << "] = " << lit(sp(k, 0)) << " * wdot[" << k << "] * invrho;\n";
  o
    << "  f[0] = -(Hw * invrho * invcp);\n"
    << "  if (WITH_J) {\n"
    << "    const double Wbar = 1.0 / sumYW;\n"
    // row k holds S'_kl = (W_k / W_l) dwdot_k/dC_l; with s_k = sum_l S_kl C_l =
    // (1 / W_k) sum_l S'_kl rho Y_l and a_k = W_k Wbar (wdot_k - s_k) / rho:
    // dY_k/dY_l = S'_kl + a_k / W_l
    << "    double rY[NS];\n#pragma unroll\n    for (int l = 0; l < NS; ++l) rY[l] = rho * y[1 + l];\n"
    << "#pragma unroll 1\n"
    << "    for (int k = 0; k < NS; ++k) {\n"
    << "      const int row = (1 + k) * n;\n      const double Wk = mv.sp[SP_REC * k];\n"
    << "      double s = 0.0;\n#pragma unroll\n      for (int l = 0; l < NS; ++l) s += Jv[row + 1 + l] * rY[l];\n"
    << "      s = s * mv.sp[SP_REC * k + 1];\n"
    << (any_collider ? "      const double sMk = sM[k];\n      s = fma(sMk, ctot, s);\n" : "")
    << "      const double wk = wdot[k];\n      double a = Wk * Wbar * invrho * (wk - s);\n"
    << (any_collider ? "      a = fma(Wk, sMk, a);\n" : "")
    << "#pragma unroll\n      for (int i = 0; i < NS; ++i) Jv[row + 1 + i] = fma(a, mv.sp[SP_REC * i + 1], Jv[row + 1 + i]);\n"
    << "      Jv[row] = Wk * invrho * (Jv[row] + (wk - s) * invT);\n    }\n"
    << "    double dcp = 0.0, cpf = 0.0;\n";
  for (int k = 0; k < N; ++k) {
    const std::vector<double> d = {sp(k, 3), 2.0 * sp(k, 4), 3.0 * sp(k, 5), 4.0 * sp(k, 6)};
    o << "    dcp += y[" << 1 + k << "] * (" << horner(d, "T") << ") * " << lit(sp(k, 1)) << ";\n"
      << "    cpf += cpW[" << k << "] * f[" << 1 + k << "];\n";
  }
  o
    << "    dcp = dcp * RU;\n    cpf = cpf * RU;\n"
    // the temperature row's species weights (h_k/RT) / W_k, once
    << "    double hw[NS];\n";
  for (int k = 0; k < N; ++k) o << "    hw[" << k << "] = hRT[" << k << "] * " << lit(sp(k, 1)) << ";\n";
  o
    << "#pragma unroll 1\n    for (int jc = 0; jc < n; ++jc) {\n      double acc = 0.0;\n"
    << "#pragma unroll\n      for (int k = 0; k < NS; ++k) acc += hw[k] * Jv[(1 + k) * n + jc];\n"
    << "      acc = acc * (RU * T);\n"
    << "      if (jc == 0) {\n        Jv[0] = -(invcp * (acc + cpf)) - f[0] * dcp * invcp;\n      } else {\n"
    << "        const double cpj = RU * cpW[jc - 1];\n"
    << "        Jv[jc] = -(invcp * acc) - f[0] * cpj * invcp;\n      }\n    }\n  }\n"
    << "  return -Hw;\n}\n\n";
}

// ---------------------------------------------------------------------------
// the fixed-point evaluation
// ---------------------------------------------------------------------------

std::string hex64(uint64_t v) {
  char b[32];
  snprintf(b, sizeof b, "0x%llxull", (unsigned long long)v);
  return b;
}

// "+= c * mono" in units of 2^-bits, mono a fixed-point variable of the given scale
std::string fixed_term(const std::string& dst, double c, bool log2e, const char* mono, int scale, int bits = 53) {
  uint64_t l;
  int sh;
  fixed_literal(c, log2e, bits + 64 - scale, &l, &sh);
  if (l == 0) return "";
  std::string e = std::string("mul_fixed(") + mono + ", " + hex64(l) + ")";
  if (sh) e = "(" + e + " << " + std::to_string(sh) + ")";
  return "    " + dst + (c < 0.0 ? " -= " : " += ") + "(int64_t)" + e + ";\n";
}

// c, or c log2(e), in units of 2^-bits
std::string fixed_const(double c, bool log2e, int bits = 53) {
  uint64_t l;
  int sh;
  fixed_literal(c, log2e, bits, &l, &sh);
  return std::string(c < 0.0 ? "-" : "") + "(int64_t)(" + hex64(l) + (sh ? " << " + std::to_string(sh) : "") + ")";
}

// The fraction bits, at most 53, with which c0 + T (c1 + T (c2 + T (c3 + T c4))) + c5/T
// stays within 63 bits at the temperatures from T_low (sampled as in fixed_T_low; a
// term may wrap, the sum of 64-bit words is the same)
int enthalpy_bits(const std::vector<double>& c, double T_low) {
  double worst = 0.0;
  for (double T = T_low; T < FIX_T_HIGH * 1.02; T *= 1.02)
    worst = std::max(worst, std::fabs(c[0] + T * (c[1] + T * (c[2] + T * (c[3] + T * c[4]))) + c[5] / T));
  int bits = 53;
  while (bits > 0 && worst * 1.05 * std::ldexp(1.0, bits) >= 0x1p63) --bits;
  return bits;
}

// The unknowns of the generated kernel's linear systems.  A species that no
// reaction changes is inert.  Of the others the mole changes live in the column
// space of the stoichiometric matrix: with as many fewer dimensions as elements
// are conserved, dn_e = sum_r b_er dn_r expresses some species (elim) by the rest
// (keep), exactly, for the production rates, every stage vector of a Rosenbrock
// step and the step itself.  The systems then cover the kept species and the
// temperature.  Eliminated are molecules of non-positive formation enthalpy (the
// species that carry the mass, so that a sum's rounding is small beside them)
// with the most reactions (whose production rates need not be summed).
struct Systems {
  std::vector<int> act;    // reacting species, ascending
  std::vector<int> keep;   // species of the systems' rows, ascending
  std::vector<int> elim;   // eliminated species, ascending
  std::vector<std::vector<double>> b;  // [elim][keep]
  int na() const { return (int)keep.size() + 1; }
  // doubles of shared memory per thread: the matrix and a vector, or the kept
  // species' rows over all reacting species while the Jacobian is summed
  int per_thread() const {
    return std::max(na() * (na() + 1), (int)(keep.size() * (act.size() + 1)));
  }
  // further words, for the exponents of a group of reactions.  More words make
  // longer runs of independent work, but what shared memory does not take is L1 for
  // the threads' local memory (states, stage vectors): 2^20 cells of the 9-species
  // field take 16.6, 15.9, 16.1, 16.9, 18.6 ms with 12, 20, 28, 36, 52 words.
  static constexpr int exponents() { return 20; }
};

struct Ratio {
  long long p = 0, q = 1;
};
bool ratio_sub_mul(Ratio* a, Ratio f, Ratio x) {  // a -= f x; false on overflow
  long long p, q, u, v, w;
  if (__builtin_mul_overflow(f.p, x.p, &p) || __builtin_mul_overflow(f.q, x.q, &q) ||
      __builtin_mul_overflow(a->p, q, &u) || __builtin_mul_overflow(p, a->q, &v) || __builtin_sub_overflow(u, v, &w) ||
      __builtin_mul_overflow(a->q, q, &q))
    return false;
  const long long g = std::max(1ll, std::__gcd(w < 0 ? -w : w, q < 0 ? -q : q));
  a->p = w / g;
  a->q = q / g;
  return true;
}

Systems systems_of(const df_mech* m, const std::vector<Rx>& rx) {
  const int N = m->dims.N, M = (int)rx.size();
  Systems s;
  std::vector<int> entries(N, 0);
  for (int k = 0; k < N; ++k) {
    for (const Rx& x : rx) entries[k] += x.nu[k] != 0;
    if (entries[k]) s.act.push_back(k);
  }
  auto stable = [&](int k) {  // h(298 K)
    const double* a = &m->blob_host[m->dims.off_sp + SP_REC * k + 2];
    const double T = 298.0;
    return a[0] * T + T * T * (a[1] / 2 + T * (a[2] / 3 + T * (a[3] / 4 + T * a[4] / 5))) + a[5] <= 1500.0;
  };
  std::vector<int> order = s.act;  // the last ones that depend on the earlier ones are eliminated
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) {
    return std::make_pair(stable(a), entries[a]) < std::make_pair(stable(b), entries[b]);
  });
  // row echelon form of the kept species' rows, each with its combination of them
  struct Row {
    std::vector<Ratio> v;   // M entries
    std::vector<Ratio> c;   // by position in `kept`
    int pivot;
  };
  std::vector<Row> basis;
  std::vector<int> kept;
  std::vector<std::pair<int, std::vector<Ratio>>> dep;
  bool ok = true;
  for (int k : order) {
    Row r;
    r.v.resize(M);
    for (int j = 0; j < M; ++j) r.v[j].p = rx[j].nu[k];
    r.c.assign(order.size(), Ratio());
    for (const Row& e : basis) {
      if (r.v[e.pivot].p == 0) continue;
      Ratio f{r.v[e.pivot].p * e.v[e.pivot].q, r.v[e.pivot].q * e.v[e.pivot].p};
      if (f.q < 0) f = Ratio{-f.p, -f.q};
      for (int j = 0; j < M && ok; ++j) ok = ratio_sub_mul(&r.v[j], f, e.v[j]);
      for (size_t i = 0; i < r.c.size() && ok; ++i) ok = ratio_sub_mul(&r.c[i], f, e.c[i]);
    }
    if (!ok) break;
    r.pivot = -1;
    for (int j = 0; j < M && r.pivot < 0; ++j)
      if (r.v[j].p != 0) r.pivot = j;
    if (r.pivot < 0) {
      dep.emplace_back(k, r.c);  // nu_k + sum_i c_i nu_kept[i] = 0
    } else {
      r.c[kept.size()].p += 1;
      kept.push_back(k);
      basis.push_back(r);
    }
  }
  if (!ok) {  // no elimination
    s.keep = s.act;
    return s;
  }
  s.keep = kept;
  std::sort(s.keep.begin(), s.keep.end());
  std::sort(dep.begin(), dep.end(), [](const auto& a, const auto& b) { return a.first < b.first; });
  for (const auto& d : dep) {
    s.elim.push_back(d.first);
    std::vector<double> b;
    for (int k : s.keep) {
      const Ratio c = d.second[std::find(kept.begin(), kept.end(), k) - kept.begin()];
      b.push_back(-(double)c.p / (double)c.q + 0.0);
    }
    s.b.push_back(b);
  }
  return s;
}

// The product of the rate constant `K` and the concentrations C[e], unpacked: `name`p,
// and with derivatives by each distinct species the doubles `name`d<l>; `name`s is
// the sign word of the product
std::string fx_product_code(const std::string& name, const std::string& K, std::vector<int> e, bool deriv) {
  std::ostringstream o;
  auto X = [](int k) { return "x" + std::to_string(k); };
  auto hi = [](int k) { return "(uint32_t)__double2hiint(C[" + std::to_string(k) + "])"; };
  auto sgn = [&](std::vector<int> v) {
    std::string s;
    for (int k : v) s += (s.empty() ? "" : " ^ ") + hi(k);
    return s.empty() ? std::string("0u") : s;
  };
  auto mul = [](const std::string& a, const std::string& b) { return "fx_mul(" + a + ", " + b + ")"; };
  if (e.size() == 3 && e[0] != e[1]) {  // equal species first
    if (e[0] == e[2]) std::swap(e[1], e[2]);
    else if (e[1] == e[2]) std::swap(e[0], e[2]);
  }
  o << "    const uint32_t " << name << "s = " << sgn(e) << ";\n";
  if (!deriv) {
    std::string p = K;
    for (int k : e) p = mul(p, X(k));
    o << "    const Fx " << name << "p = " << p << ";\n";
    return o.str();
  }
  auto fx = [&](const char* v, const std::string& x) { o << "    const Fx " << name << v << " = " << x << ";\n"; };
  // d/dC_l = mult v, v an unpacked number with the sign of the other species
  auto d = [&](int l, int mult, const std::string& v, std::vector<int> others) {
    const std::string p = "fx_pack(" + v + (mult == 2 ? ".m, " + v + ".e + 1" : std::string()) + ", " + sgn(others) + ")";
    o << "    const double " << name << "d" << l << " = " << (mult == 3 ? "3.0 * " : "") << p << ";\n";
  };
  if (e.size() == 1) {
    fx("t", K);
    d(e[0], 1, name + "t", {});
    fx("p", mul(name + "t", X(e[0])));
  } else if (e.size() == 2 && e[0] == e[1]) {
    fx("t", mul(K, X(e[0])));
    d(e[0], 2, name + "t", {e[0]});
    fx("p", mul(name + "t", X(e[0])));
  } else if (e.size() == 2) {
    fx("t", mul(K, X(e[0])));
    fx("u", mul(K, X(e[1])));
    d(e[1], 1, name + "t", {e[0]});
    d(e[0], 1, name + "u", {e[1]});
    fx("p", mul(name + "t", X(e[1])));
  } else if (e[0] == e[1] && e[1] == e[2]) {
    fx("t", mul(mul(K, X(e[0])), X(e[0])));
    d(e[0], 3, name + "t", {e[0], e[0]});
    fx("p", mul(name + "t", X(e[0])));
  } else if (e[0] == e[1]) {
    fx("t", mul(K, X(e[0])));
    fx("u", mul(name + "t", X(e[0])));
    fx("v", mul(name + "t", X(e[2])));
    d(e[2], 1, name + "u", {e[0], e[0]});
    d(e[0], 2, name + "v", {e[0], e[2]});
    fx("p", mul(name + "u", X(e[2])));
  } else {
    fx("t", mul(K, X(e[0])));
    fx("u", mul(name + "t", X(e[1])));
    fx("v", mul(name + "t", X(e[2])));
    fx("y", mul(mul(K, X(e[1])), X(e[2])));
    d(e[2], 1, name + "u", {e[0], e[1]});
    d(e[1], 1, name + "v", {e[0], e[2]});
    d(e[0], 1, name + "y", {e[1], e[2]});
    fx("p", mul(name + "u", X(e[2])));
  }
  return o.str();
}

// Where two products meet in a sum the text says which one is fused, so that the
// module's kernels, compiled apart, round alike.
//
// The evaluation the generated kernel runs: f and -J, the latter over the kept
// species and the temperature (Systems).  The exponents of the rate constants -- ln A + b ln T - E/T, the
// sums of g_k/RT and the pressure term, all times log2(e) -- are 64-bit
// fixed-point sums in units of 2^-53 octave: an addition is two integer
// instructions where an FP64 one occupies the pipe for 64 cycles, a product
// about a quarter of one, and the result is the argument exp2_fixed wants, more
// accurate than the rounded FP64 sums it replaces.  Only what multiplies
// concentrations stays in FP64.  Returns false (nothing written) for states
// outside the range the fixed-point words cover; the caller then takes gen_eval.
// Without J only the kept species' entries of f and f[0] are written.
void emit_fixed(std::ostringstream& o, const df_mech* m, const std::vector<Rx>& rx, const Systems& sys, double T_low,
                bool saturates) {
  const int N = m->dims.N, NA = sys.na(), NR = NA - 1, wid = (int)sys.act.size() + 1;
  auto sp = [&](int k, int i) { return m->blob_host[m->dims.off_sp + SP_REC * k + i]; };
  std::vector<int> col(N, -1), row(N, -1);  // reacting species -> column while J is summed; kept species -> row
  for (size_t a = 0; a < sys.act.size(); ++a) col[sys.act[a]] = (int)a + 1;
  for (int a = 0; a < NR; ++a) row[sys.keep[a]] = a;
  // d Y_elim[e] / d Y_keep[a]
  auto beta = [&](size_t e, int a) { return sys.b[e][a] * (sp(sys.elim[e], 0) * sp(sys.keep[a], 1)); };
  auto S = [](int k) { return std::to_string(k); };
  // the sums: a row per kept species, d/dT and the reacting species (column 0 and
  // col); then, in place row by row, the matrix, the temperature last
  auto W = [&](int a, int b) { return "W[" + std::to_string(a * wid + b) + "]"; };
  auto Wn = [&](int a, int b) { return "W[" + std::to_string(a * NA + b) + "]"; };
  bool any_collider = false, any_inert = false;  // any_inert: a rate depends on an inert species alone
  std::vector<bool> used(N, false);  // species whose g/RT some reaction needs
  for (const Rx& x : rx) {
    any_collider = any_collider || x.type != 0;
    for (int k : x.spc) {
      if (x.nu[k] != 0) used[k] = true;
      if (col[k] < 0) any_inert = true;
    }
    for (int l = 0; l < N; ++l)
      if (x.type != 0 && col[l] < 0 && m->blob_host[m->dims.off_eff + N * x.eff + l] != 1.0) any_inert = true;
  }
  // the constants of reactions without a rate: words that pack to zero in every product
  // (a call, which costs nothing where it is not made: 2^20 cells 15.5 ms, inlined 16.2)
  o << "template <int ST>\n"
    << "__device__ __noinline__ void gen_no_rate(const MechView& mv, int j0, int j1, SVT<double, ST> E) {\n"
    << "  int at = 0;\n"
    << "#pragma unroll 1\n  for (int j = j0; j < j1; ++j) {\n"
    << "    const RxMeta mt = load_meta(mv.rx + RX_REC * j);\n"
    << "    const int words = 1 + ((mt.flags & 3) == 2 ? 1 : 0) + ((mt.flags & 4) != 0 ? 1 : 0);\n"
    << "    if (mv.fix[j] == FIX_OFF)\n"
    << "      for (int i = 0; i < words; ++i) E[at + i] = 0.0;\n"
    << "    at += words;\n  }\n}\n\n";
  o << "template <bool WITH_J, int ST>\n"
    << "__device__ __forceinline__ bool gen_fixed(const MechView& mv, const double pc, const double (&y)[" << N + 1
    << "], double (&f)[" << N + 1 << "], SVT<double, ST> W, SVT<double, ST> E) {\n"
    << "  constexpr int NS = " << N << ";\n"
    << "  const double T = y[0];\n"
    << "  const long long flag = mv.fix[" << m->dims.M << "];\n"
    << "  if (!flag || !(T >= " << lit(T_low) << " && T < " << lit(FIX_T_HIGH) << ")) return false;\n"
    << "  double C[NS], cpW[NS];  // cpW: cp_k / (R W_k)\n"
    << "  double sumYW = 0.0, cpm = 0.0;\n";
  for (int k = 0; k < N; ++k) {
    std::vector<double> aw = {sp(k, 2), sp(k, 3), sp(k, 4), sp(k, 5), sp(k, 6)};
    for (double& v : aw) v *= sp(k, 1);
    o << "  C[" << k << "] = y[" << 1 + k << "] * " << lit(sp(k, 1)) << ";\n  sumYW += C[" << k << "];\n"
      << "  cpW[" << k << "] = " << horner(aw, "T") << ";\n  cpm += y[" << 1 + k << "] * cpW[" << k << "];\n";
  }
  o << "  if (!rcp_in_range(sumYW) || !rcp_in_range(cpm) || !rcp_in_range(pc)) return false;\n"
    // (cpm RU, 2^26 times cpm, is within what rcp_fast takes: below 2^124)
    << "  const double invT = rcp_fast(T), Wbar = rcp_fast(sumYW), invcp = rcp_fast(cpm * RU);\n"
    << "  const double rho = pc * invT * (Wbar * " << lit(1.0 / RU) << ");\n"
    << "  const double invrho = rcp_any(rho);\n"
    << "  // log2 T, 1/T, T and its powers in fixed point\n"
    << "  const uint64_t L = log2_fixed(T), I = pos_fixed<69>(invT), t1 = pos_fixed<50>(T);\n"
    << "  const uint64_t t2 = mul_fixed(t1, t1);\n";
  bool t3 = false, t4 = false;
  for (int k = 0; k < N; ++k) {
    t3 = t3 || ((used[k] || col[k] > 0) && sp(k, 5) != 0.0);
    t4 = t4 || ((used[k] || col[k] > 0) && sp(k, 6) != 0.0);
  }
  if (t3) o << "  const uint64_t t3 = mul_fixed(t2, t1);\n";
  if (t4) o << "  const uint64_t t4 = mul_fixed(t2, t2);\n";
  o << "  const int64_t lp = " << fixed_const(LOG_PSTD_RU, true) << " - (int64_t)(L >> 7);  // log2(p_std / (R T))\n"
    << "  int64_t G[NS];  // g_k/RT log2(e)\n";
  for (int k = 0; k < N; ++k) {
    if (!used[k]) continue;
    const std::string g = "G[" + S(k) + "]";
    o << "  {\n    " << g << " = " << fixed_const(sp(k, 2) - sp(k, 8), true) << ";\n"
      << fixed_term(g, -sp(k, 2), false, "L", 60) << fixed_term(g, -0.5 * sp(k, 3), true, "t1", 50)
      << fixed_term(g, -sp(k, 4) / 6.0, true, "t2", 36) << fixed_term(g, -sp(k, 5) / 12.0, true, "t3", 22)
      << fixed_term(g, -sp(k, 6) / 20.0, true, "t4", 8) << fixed_term(g, sp(k, 7), true, "I", 69) << "  }\n";
  }
  for (int k = 0; k < N; ++k) o << "  C[" << k << "] *= rho;\n";
  if (any_collider) {
    o << "  const double ctot = rho * sumYW;\n";
  }
  for (int k = 0; k < N; ++k) o << "  const Fx x" << k << " = fx_factor(C[" << k << "]);\n  (void)x" << k << ";\n";
  // h/RT: with J of every reacting species, in fixed point, for d ln K_c/dT
  o << "  double w[NS], sM[NS], sN[NS];\n  int64_t H[NS];\n  (void)H; (void)sM; (void)sN;\n";
  auto enthalpy = [&](const std::string& dst, const std::vector<double>& c, int bits) {
    return "    " + dst + " = " + fixed_const(c[0], false, bits) + ";\n" + fixed_term(dst, c[1], false, "t1", 50, bits) +
           fixed_term(dst, c[2], false, "t2", 36, bits) + fixed_term(dst, c[3], false, "t3", 22, bits) +
           fixed_term(dst, c[4], false, "t4", 8, bits) + fixed_term(dst, c[5], false, "I", 69, bits);
  };
  auto hcoef = [&](int k) {
    return std::vector<double>{sp(k, 2), sp(k, SP_H), sp(k, SP_H + 1), sp(k, SP_H + 2), sp(k, SP_H + 3), sp(k, 7)};
  };
  o << "  if (WITH_J) {\n";
  for (int k : sys.act) o << enthalpy("H[" + S(k) + "]", hcoef(k), 53);
  o << "  }\n";
  // accumulators start at zero where their first contribution is conditional
  // (falloff reactions without a low-pressure rate contribute nothing)
  std::vector<bool> w_set(N, false), sM_set(N, false), W_set(NR * wid, false);
  {
    std::vector<bool> wz(N, true), Wz(NR * wid, true), sMz(N, true);
    std::vector<bool> seen_w(N, false), seen_W(NR * wid, false), seen_M(N, false);
    for (const Rx& x : rx) {
      for (int k : x.spc) {
        const int a = row[k];
        if (x.nu[k] == 0 || a < 0) continue;
        if (!seen_w[k]) wz[k] = x.type == 2;
        seen_w[k] = true;
        if (x.type != 0) {
          if (!seen_M[k]) sMz[k] = x.type == 2;
          seen_M[k] = true;
        }
        std::vector<int> cols = {0};
        for (int l : x.spc)
          if (col[l] > 0 && (x.rev || std::find(x.r.begin(), x.r.end(), l) != x.r.end())) cols.push_back(col[l]);
        for (int c : cols) {
          if (!seen_W[a * wid + c]) Wz[a * wid + c] = x.type == 2;
          seen_W[a * wid + c] = true;
        }
        if (x.type != 0)
          for (int l = 0; l < N; ++l)
            if (m->blob_host[m->dims.off_eff + N * x.eff + l] != 1.0 && col[l] > 0) {
              const int c = col[l];
              if (!seen_W[a * wid + c]) Wz[a * wid + c] = true;
              seen_W[a * wid + c] = true;
            }
      }
    }
    for (int k : sys.keep) {
      if (wz[k]) {
        o << "  w[" << k << "] = 0.0;\n";
        w_set[k] = true;
      }
      if (any_collider && sMz[k]) {
        o << "  if (WITH_J) sM[" << k << "] = 0.0;\n";
        sM_set[k] = true;
      }
      if (any_inert) o << "  if (WITH_J) sN[" << k << "] = 0.0;\n";
    }
    o << "  if (WITH_J) {\n";
    for (int a = 0; a < NR; ++a)
      for (int b = 0; b < wid; ++b)
        if (Wz[a * wid + b]) {
          o << "    " << W(a, b) << " = 0.0;\n";
          W_set[a * wid + b] = true;
        }
    o << "  }\n";
  }
  // the rows take -d w_k/d(...) , species columns pre-scaled by W_k / W_l
  auto addW = [&](int a, int b, double c, const std::string& v) {
    std::ostringstream s;
    const bool set = W_set[a * wid + b];
    W_set[a * wid + b] = true;
    s << "      " << W(a, b);
    if (c == 1.0) s << (set ? " -= " : " = -") << v << ";\n";
    else if (c == -1.0) s << (set ? " += " : " = ") << v << ";\n";
    else s << (set ? " -= " : " = -") << lit(c) << " * " << v << ";\n";
    return s.str();
  };
  auto add1 = [&](std::vector<bool>& set, const char* arr, int k, int c, const std::string& v) {
    std::ostringstream s;
    s << arr << "[" << k << "]";
    const bool st = set[k];
    set[k] = true;
    if (c == 1) s << (st ? " += " : " = ") << v << ";\n";
    else if (c == -1) s << (st ? " -= " : " = -") << v << ";\n";
    else s << (st ? " += " : " = ") << c << ".0 * " << v << ";\n";
    return s.str();
  };
  // the exponents of the reactions [j, j1) and then all their powers of two: of an
  // elementary or third-body reaction k_f and (reversible) k_r, of a falloff
  // reaction k_inf, k_0 / k_inf and (reversible) 1 / K_c
  const int cap = Systems::exponents();
  std::vector<int> slot(rx.size());
  auto exponents = [&](size_t j0) {
    size_t j1 = j0;
    int n = 0;
    for (; j1 < rx.size(); ++j1) {
      const int words = 1 + (rx[j1].type == 2 ? 1 : 0) + (rx[j1].rev ? 1 : 0);
      if (n + words > cap) break;
      slot[j1] = n;
      n += words;
    }
    auto E = [&](int i) { return "    E[" + std::to_string(i) + "] = __longlong_as_double("; };
    for (size_t j = j0; j < j1; ++j) {
      const Rx& x = rx[j];
      o << "  {\n    int64_t x = mv.fix[" << j << "];\n"
        << fixed_term("x", x.b, false, "L", 60) << fixed_term("x", -x.E, true, "I", 69) << E(slot[j]) << "x);\n";
      std::string sg;
      for (int k : x.spc)
        for (int i = 0; i < std::abs(x.nu[k]); ++i) sg += (x.nu[k] > 0 ? " + G[" : " - G[") + S(k) + "]";
      for (int i = 0; i < std::abs(x.dnu); ++i) sg += x.dnu > 0 ? " - lp" : " + lp";
      if (x.type == 2) {
        const double* tr = &m->blob_host[m->dims.off_tr + TR_REC * x.troe];
        o << "    int64_t xd = " << fixed_const(tr[0] == -INFINITY ? 0.0 : tr[0], true) << ";\n"
          << fixed_term("xd", tr[1] - x.b, false, "L", 60) << fixed_term("xd", -(tr[2] - x.E), true, "I", 69)
          << E(slot[j] + 1) << "xd);\n";
        if (x.rev) o << E(slot[j] + 2) << "(int64_t)0" << sg << ");\n";
      } else if (x.rev) {
        o << E(slot[j] + 1) << (saturates ? "add_exponents(x, (int64_t)0" + sg + ")" : "x" + sg) << ");\n";
      }
      o << "  }\n";
    }
    const int padded = (n + 3) / 4 * 4;
    for (int i = n; i < padded; ++i) o << E(i).substr(2) << "0);\n";
    o << "  fx_exp2_all<" << padded << ">(E);\n"
      << "  if (flag == 2) gen_no_rate(mv, " << j0 << ", " << j1 << ", E);\n";
    return j1;
  };
  size_t group_end = 0;
  for (size_t j = 0; j < rx.size(); ++j) {
    const Rx& x = rx[j];
    if (j == group_end) group_end = exponents(j);
    auto K = [&](int i) { return "fx_word(E[" + std::to_string(i) + "])"; };
    o << "  {  // rate " << j << "\n";
    if (x.type != 0) {
      o << "    double Mc = ctot;\n";
      for (int l = 0; l < N; ++l) {
        const double e = m->blob_host[m->dims.off_eff + N * x.eff + l];
        if (e != 1.0) o << "    Mc += " << lit(e - 1.0) << " * C[" << l << "];\n";
      }
    }
    // d ln k / dT and d ln K_c / dT
    std::ostringstream dl;
    // (times T: the column d/dT takes the factor 1/T when the row is finished)
    dl << "      int64_t bE = " << fixed_const(x.b, false) << ";\n"
       << fixed_term("bE", x.E, false, "I", 69) << "      const double dk = fixed_to_double(bE);\n";
    std::string dKc = "fixed_to_double(" + S(-x.dnu) + "LL * (1LL << 53)";
    for (int k : x.spc)
      for (int i = 0; i < std::abs(x.nu[k]); ++i) dKc += (x.nu[k] > 0 ? " + H[" : " - H[") + S(k) + "]";
    dKc += ")";
    auto has_dq = [&](int l) {
      return std::find(x.r.begin(), x.r.end(), l) != x.r.end() ||
             (x.rev && std::find(x.p.begin(), x.p.end(), l) != x.p.end());
    };
    // the Jacobian rows from dq<l>, dqT and, with a collider, dqM
    auto rows = [&]() {
      std::ostringstream s;
      for (int k : x.spc) {
        const int a = row[k];
        if (x.nu[k] == 0 || a < 0) continue;
        s << addW(a, 0, x.nu[k], "dqT");
        for (int l : x.spc) {
          if (!has_dq(l)) continue;
          if (col[l] > 0)
            s << addW(a, col[l], l == k ? (double)x.nu[k] : x.nu[k] * (sp(k, 0) * sp(l, 1)), "dq" + S(l));
          else  // an inert species: no column, but its share of s_k
            s << "      sN[" << k << "] += " << lit(x.nu[k]) << " * (dq" << l << " * C[" << l << "]);\n";
        }
        if (x.type != 0) {
          s << "      " << add1(sM_set, "sM", k, x.nu[k], "dqM");
          for (int l = 0; l < N; ++l) {
            const double e = m->blob_host[m->dims.off_eff + N * x.eff + l];
            if (e == 1.0) continue;
            if (col[l] > 0)
              s << addW(a, col[l], x.nu[k] * (e - 1.0) * (l == k ? 1.0 : sp(k, 0) * sp(l, 1)), "dqM");
            else
              s << "      sN[" << k << "] += " << lit(x.nu[k] * (e - 1.0)) << " * (dqM * C[" << l << "]);\n";
          }
        }
      }
      return s.str();
    };
    auto dqs = [&](const char* scale) {
      std::ostringstream s;
      for (int l : x.spc) {
        if (!has_dq(l)) continue;
        const bool inr = std::find(x.r.begin(), x.r.end(), l) != x.r.end();
        const bool inp = x.rev && std::find(x.p.begin(), x.p.end(), l) != x.p.end();
        std::string e = inr && inp ? "fd" + S(l) + " - bd" + S(l) : inr ? "fd" + S(l) : inp ? "-bd" + S(l) : "0.0";
        s << "      const double dq" << l << " = " << (*scale ? std::string(scale) + " * (" + e + ")" : e) << ";\n"
          << "      (void)dq" << l << ";\n";
      }
      return s.str();
    };
    std::ostringstream upd;
    if (x.type != 2) {
      o << "    const Fx kf = " << K(slot[j]) << ";\n";
      if (x.rev) o << "    const Fx kr = " << K(slot[j] + 1) << ";\n";
      for (int wj = 1; wj >= 0; --wj) {
        if (wj) o << "    if (WITH_J) {\n";
        else o << "    } else {\n";
        const auto w0 = w_set;  // both branches start from the same accumulators
        o << fx_product_code("f", "kf", x.r, wj);
        if (x.rev) o << fx_product_code("b", "kr", x.p, wj);
        const std::string q0 = x.rev ? "fx_diff(fp, fs, bp, bs)" : "fx_pack(fp, fs)";
        if (x.type == 1) o << "      const double dqM = " << q0 << ";\n      (void)dqM;\n      const double q = Mc * dqM;\n";
        else o << "      const double q = " << q0 << ";\n";
        for (int k : x.spc)
          if (x.nu[k] != 0 && row[k] >= 0) o << "      " << add1(w_set, "w", k, x.nu[k], "q");
        if (wj) {
          o << dl.str();
          if (x.rev) o << "      const double dKc = " << dKc << ", pb = fx_pack(bp, bs);\n";
          if (!x.rev) o << "      const double dqT = q * dk;\n";
          else if (x.type == 1) o << "      const double dqT = fma(q, dk, (Mc * pb) * dKc);\n";
          else o << "      const double dqT = fma(q, dk, pb * dKc);\n";
          o << dqs(x.type == 1 ? "Mc" : "") << rows();
          w_set = w0;  // the other branch makes the same first updates of w
        }
      }
      o << "    }\n  }\n";
      continue;
    }
    // Troe falloff: the expressions of rate_compute with logarithms to base 2, in
    // fixed point up to the quotient; k = k_inf Pr/(1 + Pr) F as an unpacked number
    const double* tr = &m->blob_host[m->dims.off_tr + TR_REC * x.troe];
    uint64_t c67, c127, c14;
    int none;
    fixed_literal(0.67, false, 64, &c67, &none);
    fixed_literal(1.27, false, 63, &c127, &none);
    fixed_literal(0.14, false, 64, &c14, &none);
    const double L10 = 3.32192809488736234787;  // log2(10)
    auto q52 = [](double v) { return std::to_string((long long)std::llround(std::ldexp(v, 52))) + "LL"; };
    o << "    const Fx kinf = " << K(slot[j]) << ";\n"
      << "    const double Pr = fx_pack(" << K(slot[j] + 1) << ", 0u) * Mc;\n"
      << "    if (Pr >= 0x1p-1022) {\n"
      << "      double e3, e1;\n      exp_rate2(-T * " << lit(tr[4]) << ", -T * " << lit(tr[5]) << ", e3, e1);\n"
      << "      const double e2 = exp_rate(" << lit(-tr[6]) << " * invT);\n"
      << "      const double Fc = fma(" << lit(1.0 - tr[3]) << ", e3, fma(" << lit(tr[3]) << ", e1, e2));\n"
      << "      const int64_t lc = log2_q52(Fc), lx = log2_q52(Pr) - " << q52(0.4 * L10) << " - mul_fixed_signed(lc, "
      << hex64(c67) << ");\n"
      << "      const int64_t ln = " << q52(0.75 * L10) << " - 2 * mul_fixed_signed(lc, " << hex64(c127) << ");\n"
      << "      const double xl = q52_to_double(lx), den = q52_to_double(ln - mul_fixed_signed(lx, " << hex64(c14) << "));\n"
      << "      const double Lc = q52_to_double(lc), den2 = den * den;\n"
      << "      const double q1 = den2 * rcp_any(fma(xl, xl, den2)), onePr = rcp_any(1.0 + Pr);\n"
      << "      const Fx kf = fx_mul(fx_mul(kinf, fx_factor(Pr * onePr)), fx_exp2_factor(Lc * q1));\n";
    if (x.rev) {
      o << "      Fx kr = " << K(slot[j] + 2) << ";\n      kr.e += 64;\n      kr = fx_mul(kf, kr);\n";
    }
    for (int wj = 1; wj >= 0; --wj) {
      const auto w0 = w_set;
      o << (wj ? "      if (WITH_J) {\n" : "      } else {\n") << fx_product_code("f", "kf", x.r, wj);
      if (x.rev) o << fx_product_code("b", "kr", x.p, wj);
      o << "      const double q = " << (x.rev ? "fx_diff(fp, fs, bp, bs)" : "fx_pack(fp, fs)") << ";\n";
      for (int k : x.spc)
        if (x.nu[k] != 0 && row[k] >= 0) o << "      " << add1(w_set, "w", k, x.nu[k], "q");
      if (wj) {
        o << "      const double nn = q52_to_double(ln), rden = rcp_any(den), f1 = xl * rden;\n"
          << "      const double df1_dL = nn * rden * rden;\n"
          << "      const double df1_dLc = fma(-0.67, den, -(xl * (-1.27 + 0.67 * 0.14))) * (rden * rden);\n"
          << "      const double g2 = 2.0 * Lc * f1 * q1 * q1;\n"
          << "      const double gpr = fma(-g2, df1_dL, onePr), dlogF_dLc = fma(-g2, df1_dLc, q1);\n"
          << "      const double dFc = fma(T, fma(" << lit(-(1.0 - tr[3]) * tr[4]) << ", e3, " << lit(-tr[3] * tr[5])
          << " * e1), " << lit(tr[6]) << " * (invT * e2));\n"
          << "      const double dki = fma(" << lit(x.E) << ", invT, " << lit(x.b) << ");\n"
          << "      const double dk0 = fma(" << lit(tr[2]) << ", invT, " << lit(tr[1]) << ");\n"
          << "      const double dk = fma(dlogF_dLc * dFc, rcp_any(Fc), fma(gpr, dk0 - dki, dki));\n";
        if (x.rev)
          o << "      const double dKc = " << dKc << ", pb = fx_pack(bp, bs);\n"
            << "      const double dqT = fma(q, dk, pb * dKc);\n";
        else
          o << "      const double dqT = q * dk;\n";
        // dk/d[M] = k gpr / [M]
        o << "      const double dqM = q * (gpr * rcp_any(Mc));\n" << dqs("") << rows();
        w_set = w0;
      }
    }
    o << "      }\n    }\n  }\n";
  }
  // h/RT of the kept species with the eliminated ones' shares (the heat release
  // and the temperature row need no others).  A fuel's is its heat of combustion, so
  // beyond 1024 a sum has fewer fraction bits than 53 (still more digits than a double)
  o << "  double hk[NS];\n";
  for (int a = 0; a < NR; ++a) {
    std::vector<double> c = hcoef(sys.keep[a]);
    for (size_t e = 0; e < sys.elim.size(); ++e) {
      const std::vector<double> ce = hcoef(sys.elim[e]);
      for (int i = 0; i < 6; ++i) c[i] += sys.b[e][a] * ce[i];
    }
    const int bits = enthalpy_bits(c, T_low);
    o << "  {\n    int64_t h;\n" << enthalpy("h", c, bits) << "    hk[" << sys.keep[a] << "] = fixed_to_double(h"
      << (bits != 53 ? ", " + S(bits) : std::string()) << ");\n  }\n";
  }
  // heat release and f
  o << "  double Hw = 0.0;\n";
  for (int k : sys.keep) o << "  Hw += hk[" << k << "] * w[" << k << "];\n";
  for (int k : sys.keep) o << "  f[" << 1 + k << "] = " << lit(sp(k, 0)) << " * (w[" << k << "] * invrho);\n";
  o << "  const double RT = RU * T;\n  f[0] = -(Hw * RT) * (invrho * invcp);\n  if (WITH_J) {\n";
  for (size_t e = 0; e < sys.elim.size(); ++e) {
    o << "    f[" << 1 + sys.elim[e] << "] = 0.0";
    for (int a = 0; a < NR; ++a)
      if (sys.b[e][a] != 0.0) o << " + " << lit(beta(e, a)) << " * f[" << 1 + sys.keep[a] << "]";
    o << ";\n";
  }
  for (int k = 0; k < N; ++k)
    if (col[k] < 0) o << "    f[" << 1 + k << "] = 0.0;\n";
  // -J: row k holds -S'_kl = -(W_k / W_l) dw_k/dC_l; with s_k = sum_l S_kl C_l and
  // a_k = W_k (Wbar / rho) (w_k - s_k) + W_k sM_k: d f_k/dY_l = S'_kl + a_k / W_l
  // (gen_eval); a kept species' column takes beta times the eliminated ones'; the
  // temperature row sums the finished rows
  o << "    const double wb = Wbar * invrho;\n    double dcp = 0.0, cpf = 0.0;\n";
  for (int b = 0; b < NA; ++b) o << "    double tr" << b << " = 0.0;\n";
  for (int a = 0; a < NR; ++a) {
    const int k = sys.keep[a];
    o << "    {  // row of species " << k << "\n      const double v0 = " << W(a, 0) << ";\n";
    for (int l : sys.act) o << "      const double v" << 1 + l << " = " << W(a, col[l]) << ";\n";
    o << "      double s = 0.0;\n";
    for (int l : sys.act) o << "      s -= v" << 1 + l << " * (rho * y[" << 1 + l << "]);\n";
    o << "      s = s * " << lit(sp(k, 1)) << ";\n";
    if (any_collider) o << "      s = fma(sM[" << k << "], ctot, s);\n";
    if (any_inert) o << "      s += sN[" << k << "];\n";
    o << "      const double ws = w[" << k << "] - s, hw = hk[" << k << "] * " << lit(sp(k, 1)) << ";\n"
      << "      const double ak = " << lit(sp(k, 0)) << " * (wb * ws" << (any_collider ? " + sM[" + S(k) + "]" : std::string())
      << ");\n";
    for (int b = 0; b < NR; ++b) {
      const int l = sys.keep[b];
      double iw = sp(l, 1);
      o << "      const double n" << b << " = v" << 1 + l;
      for (size_t e = 0; e < sys.elim.size(); ++e)
        if (sys.b[e][b] != 0.0) {
          o << " + " << lit(beta(e, b)) << " * v" << 1 + sys.elim[e];
          iw += beta(e, b) * sp(sys.elim[e], 1);
        }
      o << " - ak * " << lit(iw) << ";\n      " << Wn(a, b) << " = n" << b << ";\n      tr" << b << " += hw * n" << b
        << ";\n";
    }
    o << "      const double nT = " << lit(sp(k, 0)) << " * ((v0 - ws) * (invrho * invT));\n      " << Wn(a, NR)
      << " = nT;\n      tr" << NR << " += hw * nT;\n    }\n";
  }
  for (int k = 0; k < N; ++k) {
    const std::vector<double> d = {sp(k, 3), 2.0 * sp(k, 4), 3.0 * sp(k, 5), 4.0 * sp(k, 6)};
    std::vector<double> dw(d);
    for (double& v : dw) v *= sp(k, 1);
    o << "    dcp += y[" << 1 + k << "] * (" << horner(dw, "T") << ");\n";
    if (col[k] > 0) o << "    cpf += cpW[" << k << "] * f[" << 1 + k << "];\n";
  }
  o << "    const double rc = RU * invcp;\n";
  for (int b = 0; b < NR; ++b) {
    o << "    " << Wn(NR, b) << " = rc * fma(f[0], cpW[" << sys.keep[b] << "]";
    for (size_t e = 0; e < sys.elim.size(); ++e)
      if (sys.b[e][b] != 0.0) o << " + " << lit(beta(e, b)) << " * cpW[" << sys.elim[e] << "]";
    o << ", -(T * tr" << b << "));\n";
  }
  o << "    " << Wn(NR, NR) << " = rc * fma(-T, tr" << NR << ", fma(f[0], dcp, cpf));\n  }\n  return true;\n}\n\n";
}

}  // namespace

std::string jit_thread_source(const df_mech* m) {
  const int N = m->dims.N, n = N + 1;
  const std::vector<Rx> rx = reactions_of(m);
  const Systems sys = systems_of(m, rx);
  const int NA = sys.na(), NE = (int)sys.elim.size();
  // down to 300 K without the test for saturation where the mechanism allows it
  double T_low = fixed_T_low(m, rx, false);
  const bool saturates = !(T_low > 0.0 && T_low <= 300.0);
  if (saturates) T_low = fixed_T_low(m, rx, true);
  std::ostringstream o;
  o << "// generated for a " << N << "-species / " << m->dims.M << "-reaction mechanism\n"
    << "#include \"integrate_thread.cuh\"\n\nnamespace df {\n\n";
  emit_eval(o, m);
  if (T_low > 0.0) emit_fixed(o, m, rx, sys, T_low, saturates);
  std::string act, elim, beta;
  for (int k : sys.keep) act += std::to_string(1 + k) + ", ";
  for (int k : sys.elim) elim += std::to_string(1 + k) + ", ";
  for (int e = 0; e < NE; ++e) {
    beta += "{";
    for (int a = 0; a < NA; ++a) {
      const double b = a < NA - 1 ? sys.b[e][a] * (m->blob_host[m->dims.off_sp + SP_REC * sys.elim[e]] *
                                                   m->blob_host[m->dims.off_sp + SP_REC * sys.keep[a] + 1])
                                  : 0.0;
      beta += lit(b) + ", ";
    }
    beta += "}, ";
  }
  o << "struct GenEval {\n"
    << "  static constexpr bool kGenerated = true;\n"
    << "  static constexpr int kN = " << N << ", kNA = " << NA << ", kNE = " << NE << ";\n"
    << "  static constexpr int kWords = " << sys.per_thread() << ";  // shared doubles per thread before the exponents'\n"
    << "  // state entry (0: T, 1 + k: Y_k) of row a of the linear systems\n"
    << "  __device__ static constexpr int act(int a) {\n    constexpr int t[] = {" << act << "0};\n    return t[a];\n  }\n"
    << "  // state entry of eliminated species e, and d Y_e / d Y of row a\n"
    << "  __device__ static constexpr int elim(int e) {\n    constexpr int t[] = {" << elim << "0};\n    return t[e];\n  }\n"
    << "  __device__ static constexpr double beta(int e, int a) {\n    constexpr double t[][" << NA << "] = {" << beta
    << "{0.0}};\n    return t[e][a];\n  }\n"
    << "  // any state, one copy for all evaluations: the FP64 evaluation, its full\n"
    << "  // Jacobian reduced to the systems' and negated\n"
    << "  template <bool WITH_J>\n"
    << "  __device__ __noinline__ static void general(const MechView& mv, double pc, const double* y, double* f, double* W) {\n"
    << "    double yl[" << n << "], fl[" << n << "], J[WITH_J ? " << n * n << " : 1], sM[" << N << "];\n"
    << "    for (int i = 0; i < " << n << "; ++i) yl[i] = y[i];\n"
    << "    gen_eval<WITH_J, 1>(mv, pc, yl, fl, SVT<double, 1>{J, 1}, SVT<double, 1>{sM, 1});\n"
    << "    for (int i = 0; i < " << n << "; ++i) f[i] = fl[i];\n"
    << "    if (WITH_J) {\n#pragma unroll 1\n      for (int a = 0; a < kNA; ++a) {\n"
    << "#pragma unroll 1\n        for (int b = 0; b < kNA; ++b) {\n"
    << "          double v = J[act(a) * " << n << " + act(b)];\n"
    << "          for (int e = 0; e < kNE; ++e) v += beta(e, b) * J[act(a) * " << n << " + elim(e)];\n"
    << "          W[a * kNA + b] = -v;\n        }\n      }\n    }\n  }\n"
    << "  // f (without J only the entries act()) and, with WITH_J, -J over act() (row-major)\n"
    << "  template <bool WITH_J, int ST>\n"
    << "  __device__ __forceinline__ static void run(const MechView& mv, double pc, const double (&y)[" << n
    << "], double (&f)[" << n << "], SVT<double, ST> W, SVT<double, ST> E) {\n";
  if (T_low > 0.0) o << "    if (gen_fixed<WITH_J, ST>(mv, pc, y, f, W, E)) return;\n";
  o << "    double yl[" << n << "], fl[" << n << "], Wl[WITH_J ? " << NA * NA << " : 1];\n"
    << "#pragma unroll\n    for (int i = 0; i < " << n << "; ++i) yl[i] = y[i];\n"
    << "    general<WITH_J>(mv, pc, yl, fl, Wl);\n"
    << "#pragma unroll\n    for (int i = 0; i < " << n << "; ++i) f[i] = fl[i];\n"
    << "    if (WITH_J)\n#pragma unroll 1\n      for (int i = 0; i < " << NA * NA << "; ++i) W[i] = Wl[i];\n"
    << "  }\n};\n\n}  // namespace df\n";
  return o.str();
}

std::string jit_kernel_name(int N, int threads, bool ign = false) {
  return "df::k_integrate_thread<" + std::to_string(N) + ", false, " + std::to_string(threads) + ", df::GenEval" +
         (ign ? ", true>" : ">");
}

namespace {

// ---------------------------------------------------------------------------
// NVRTC (opened at run time) and the driver entry points
// ---------------------------------------------------------------------------
typedef int (*nvrtcCreateProgram_t)(void**, const char*, const char*, int, const char* const*, const char* const*);
typedef int (*nvrtcCompileProgram_t)(void*, int, const char* const*);
typedef int (*nvrtcGetSize_t)(void*, size_t*);
typedef int (*nvrtcGetBuf_t)(void*, char*);
typedef int (*nvrtcDestroyProgram_t)(void**);
typedef int (*nvrtcAddNameExpression_t)(void*, const char*);
typedef int (*nvrtcGetLoweredName_t)(void*, const char*, const char**);
typedef int (*nvrtcVersion_t)(int*, int*);

struct Nvrtc {
  bool ok = false;
  std::string why;
  nvrtcCreateProgram_t create = nullptr;
  nvrtcCompileProgram_t compile = nullptr;
  nvrtcGetSize_t log_size = nullptr, cubin_size = nullptr;
  nvrtcGetBuf_t log = nullptr, cubin = nullptr;
  nvrtcDestroyProgram_t destroy = nullptr;
  nvrtcAddNameExpression_t add_name = nullptr;
  nvrtcGetLoweredName_t lowered = nullptr;
  int version = 0;  // major * 1000 + minor
};

const Nvrtc& nvrtc() {
  static Nvrtc r;
  static std::once_flag once;
  std::call_once(once, [] {
    const char* names[] = {"libnvrtc.so.13", "libnvrtc.so", "/usr/local/cuda/lib64/libnvrtc.so.13",
                           "/usr/local/cuda/lib64/libnvrtc.so"};
    void* h = nullptr;
    for (const char* nm : names)
      if ((h = dlopen(nm, RTLD_NOW | RTLD_LOCAL))) break;
    if (!h) {
      r.why = "NVRTC library not found";
      return;
    }
    r.create = (nvrtcCreateProgram_t)dlsym(h, "nvrtcCreateProgram");
    r.compile = (nvrtcCompileProgram_t)dlsym(h, "nvrtcCompileProgram");
    r.log_size = (nvrtcGetSize_t)dlsym(h, "nvrtcGetProgramLogSize");
    r.log = (nvrtcGetBuf_t)dlsym(h, "nvrtcGetProgramLog");
    r.cubin_size = (nvrtcGetSize_t)dlsym(h, "nvrtcGetCUBINSize");
    r.cubin = (nvrtcGetBuf_t)dlsym(h, "nvrtcGetCUBIN");
    r.destroy = (nvrtcDestroyProgram_t)dlsym(h, "nvrtcDestroyProgram");
    r.add_name = (nvrtcAddNameExpression_t)dlsym(h, "nvrtcAddNameExpression");
    r.lowered = (nvrtcGetLoweredName_t)dlsym(h, "nvrtcGetLoweredName");
    r.ok = r.create && r.compile && r.log_size && r.log && r.cubin_size && r.cubin && r.destroy && r.add_name &&
           r.lowered;
    if (auto ver = (nvrtcVersion_t)dlsym(h, "nvrtcVersion")) {
      int ma = 0, mi = 0;
      if (ver(&ma, &mi) == 0) r.version = ma * 1000 + mi;
    }
    if (!r.ok) r.why = "NVRTC library lacks an entry point";
  });
  return r;
}

typedef CUresult (*cuModuleLoadData_t)(CUmodule*, const void*);
typedef CUresult (*cuModuleGetFunction_t)(CUfunction*, CUmodule, const char*);
typedef CUresult (*cuModuleGetGlobal_t)(CUdeviceptr*, size_t*, CUmodule, const char*);
typedef CUresult (*cuLaunchKernel_t)(CUfunction, unsigned, unsigned, unsigned, unsigned, unsigned, unsigned,
                                     unsigned, CUstream, void**, void**);
typedef CUresult (*cuFuncSetAttribute_t)(CUfunction, CUfunction_attribute, int);
typedef CUresult (*cuOccupancy_t)(int*, CUfunction, int, size_t);
typedef CUresult (*cuModuleUnload_t)(CUmodule);

struct Driver {
  bool ok = false;
  cuModuleLoadData_t load = nullptr;
  cuModuleUnload_t unload = nullptr;
  cuModuleGetFunction_t get_function = nullptr;
  cuModuleGetGlobal_t get_global = nullptr;
  cuLaunchKernel_t launch = nullptr;
  cuFuncSetAttribute_t set_attr = nullptr;
  cuOccupancy_t occupancy = nullptr;
};

void* entry(const char* name) {
  void* p = nullptr;
  cudaDriverEntryPointQueryResult q;
  if (cudaGetDriverEntryPointByVersion(name, &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
      q != cudaDriverEntryPointSuccess)
    return nullptr;
  return p;
}

const Driver& driver() {
  static Driver d;
  static std::once_flag once;
  std::call_once(once, [] {
    d.load = (cuModuleLoadData_t)entry("cuModuleLoadData");
    d.unload = (cuModuleUnload_t)entry("cuModuleUnload");
    d.get_function = (cuModuleGetFunction_t)entry("cuModuleGetFunction");
    d.get_global = (cuModuleGetGlobal_t)entry("cuModuleGetGlobal");
    d.launch = (cuLaunchKernel_t)entry("cuLaunchKernel");
    d.set_attr = (cuFuncSetAttribute_t)entry("cuFuncSetAttribute");
    d.occupancy = (cuOccupancy_t)entry("cuOccupancyMaxActiveBlocksPerMultiprocessor");
    d.ok = d.load && d.unload && d.get_function && d.get_global && d.launch && d.set_attr && d.occupancy;
  });
  return d;
}

// directory of the library's device headers: next to the shared library
// (<package>/_build/lib*.so -> <package>/csrc)
std::string header_dir() {
  Dl_info info;
  if (!dladdr((void*)&header_dir, &info) || !info.dli_fname) return "";
  std::string so = info.dli_fname;
  const size_t cut = so.find_last_of('/');
  if (cut == std::string::npos) return "";
  std::string dir = so.substr(0, cut);
  const size_t up = dir.find_last_of('/');
  if (up == std::string::npos) return "";
  std::string cs = dir.substr(0, up) + "/csrc";
  std::string probe = cs + "/integrate_thread.cuh";
  if (FILE* f = fopen(probe.c_str(), "r")) {
    fclose(f);
    return cs;
  }
  return "";
}

// one compiled module per (device, kernel variant, generated source), built when
// the variant is first launched: a program that uses one block size compiles one
// kernel
struct Module {
  bool ok = false;
  std::string why;
  CUmodule mod = nullptr;
  CUfunction fn = nullptr;
  size_t compile_ms = 0;
  bool from_cache = false;
  int per_thread = 0;  // doubles of shared memory per thread: the systems and the exponents
  // compiled, but not loaded or its table not uploaded (a lack of memory, say): the
  // next launches try these again, so many times
  std::vector<char> cubin;
  std::vector<std::string> lowered;
  int retries = 0;
};

std::mutex g_mu;
std::map<std::pair<int, std::string>, Module> g_modules;  // key: device * kVariants + variant, source

// the kernel variants: 32 and 64 threads per block, and 32 threads refining the
// ignition time (IntegArgs.t_ign)
constexpr int kVariants = 3, kIgnVariant = 2;
constexpr int kVariantThreads[kVariants] = {32, 64, 32};
static_assert(kVariants <= JIT_VARIANTS, "df_mech keeps one module per variant");

// ---------------------------------------------------------------------------
// on-disk cache of compiled modules: <dir>/<key>.cubin and <key>.names (the
// lowered names of the kernels and of the table), key = FNV-1a hash of the
// generated source, the device headers it includes, the target architecture
// and the NVRTC version.  Directory: $DF_JIT_CACHE ("0" disables), else
// $XDG_CACHE_HOME/df_chem_jit, else $HOME/.cache/df_chem_jit.
// ---------------------------------------------------------------------------
uint64_t fnv1a(const std::string& s, uint64_t h = 1469598103934665603ull) {
  for (unsigned char c : s) {
    h ^= c;
    h *= 1099511628211ull;
  }
  return h;
}

bool read_file(const std::string& path, std::string* out) {
  FILE* f = fopen(path.c_str(), "rb");
  if (!f) return false;
  std::string d;
  char buf[65536];
  size_t k;
  while ((k = fread(buf, 1, sizeof buf, f)) > 0) d.append(buf, k);
  const bool ok = !ferror(f);
  fclose(f);
  if (ok) *out = std::move(d);
  return ok;
}

bool write_file_atomic(const std::string& path, const std::string& data) {
  const std::string tmp = path + ".tmp" + std::to_string((unsigned long long)getpid());
  FILE* f = fopen(tmp.c_str(), "wb");
  if (!f) return false;
  const bool ok = fwrite(data.data(), 1, data.size(), f) == data.size();
  if (fclose(f) != 0 || !ok) {
    remove(tmp.c_str());
    return false;
  }
  return rename(tmp.c_str(), path.c_str()) == 0;
}

std::string cache_dir() {
  const char* e = getenv("DF_JIT_CACHE");
  std::string d;
  if (e) {
    if (!*e || std::string(e) == "0") return "";
    d = e;
  } else if (const char* x = getenv("XDG_CACHE_HOME")) {
    d = std::string(x) + "/df_chem_jit";
  } else if (const char* hm = getenv("HOME")) {
    d = std::string(hm) + "/.cache/df_chem_jit";
  } else {
    return "";
  }
  // create the directory and its parents
  for (size_t pos = 1; pos <= d.size(); ++pos)
    if (pos == d.size() || d[pos] == '/') mkdir(d.substr(0, pos).c_str(), 0755);
  return d;
}

// the device headers' contents, hashed once per process
uint64_t headers_hash(const std::string& inc) {
  static uint64_t h = 0;
  static std::once_flag once;
  std::call_once(once, [&] {
    uint64_t acc = 1469598103934665603ull;
    const char* files[] = {"integrate_thread.cuh", "rosenbrock.cuh", "chem_thread.cuh", "dev_common.cuh",
                           "exp2fix.cuh", "exp2fix_table.inc", "log2fix.cuh", "log2fix_table.inc", "dual.cuh"};
    for (const char* fn : files) {
      std::string d;
      read_file(inc + "/" + fn, &d);
      acc = fnv1a(std::string(fn) + d, acc);
    }
    h = acc;
  });
  return h;
}

// The tables to a module's constants.  The variant's first launch may lie inside a
// stream capture of the caller, where the legacy stream may not be used: a stream of
// its own that does not wait for it (and RelaxedCapture).
bool upload_tables(CUdeviceptr dst, const RosTab (&t)[2]) {
  cudaStream_t s = nullptr;
  bool ok = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking) == cudaSuccess;
  ok = ok && cudaMemcpyAsync((void*)dst, t, sizeof(t), cudaMemcpyHostToDevice, s) == cudaSuccess;
  ok = ok && cudaStreamSynchronize(s) == cudaSuccess;
  if (s) cudaStreamDestroy(s);
  return ok;
}

// resolve the kernel and the table of a loaded cubin, upload the tables
bool finish_module(Module& r, const Driver& drv, const std::vector<char>& cubin,
                   const std::vector<std::string>& lowered) {
  if (drv.load(&r.mod, cubin.data()) != CUDA_SUCCESS) {
    r.why = "cuModuleLoadData failed";
    r.mod = nullptr;
    return false;
  }
  if (lowered.size() != 2 || lowered[0].empty() || drv.get_function(&r.fn, r.mod, lowered[0].c_str()) != CUDA_SUCCESS) {
    r.why = "generated kernel not found in the module";
    drv.unload(r.mod);
    r.mod = nullptr;
    return false;
  }
  CUdeviceptr tab = 0;
  size_t tab_bytes = 0;
  if (lowered.back().empty() || drv.get_global(&tab, &tab_bytes, r.mod, lowered.back().c_str()) != CUDA_SUCCESS ||
      tab_bytes != 2 * sizeof(RosTab)) {
    r.why = "Rosenbrock table not found in the module";
    drv.unload(r.mod);
    r.mod = nullptr;
    return false;
  }
  RosTab t[2] = {make_rodas4(), make_rodas3()};
  if (!t[0].stiff_acc || !t[1].stiff_acc) {  // ros_attempt relies on it
    r.why = "Rosenbrock table not stiffly accurate";
    drv.unload(r.mod);
    r.mod = nullptr;
    return false;
  }
  if (!upload_tables(tab, t)) {
    cudaGetLastError();
    r.why = "upload of the Rosenbrock tables failed";
    drv.unload(r.mod);
    r.mod = nullptr;
    return false;
  }
  r.ok = true;
  return true;
}

// Version of the cached entries (the cubin and its lowered-name list, and what
// finish_module expects of them); raised whenever either changes.
constexpr int kCacheFormat = 4;

Module build_module(int dev, const df_mech* m, const std::string& src, int variant) {
  Module r;
  const Driver& drv = driver();
  if (!drv.ok) {
    r.why = "driver entry points for module loading unavailable";
    return r;
  }
  const std::string inc = header_dir();
  if (inc.empty()) {
    r.why = "device headers (csrc) not found next to the library";
    return r;
  }
  int major = 0, minor = 0;
  if (cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev) != cudaSuccess) {
    r.why = "device attributes unavailable";
    return r;
  }
  const Nvrtc& nv = nvrtc();
  const std::string arch = "--gpu-architecture=sm_" + std::to_string(major * 10 + minor) + "a";
  const std::vector<std::string> names = {jit_kernel_name(m->dims.N, kVariantThreads[variant], variant == kIgnVariant),
                                          "&df::c_tab"};
  const std::string incopt = "-I" + inc;
  const char* opts[] = {arch.c_str(), "-std=c++17", incopt.c_str(), "-default-device", "-lineinfo",
                        "-diag-suppress=177"};
  // the on-disk cache: keyed by the generated source, the device headers, the
  // architecture, the NVRTC version, the compile options (the include path
  // left out: a moved tree keeps its entries) and the entry format
  const std::string dir = cache_dir();
  std::string keysrc =
      src + names[0] + arch + std::to_string(nv.version) + "|format " + std::to_string(kCacheFormat);
  for (const char* o : opts)
    if (o != incopt.c_str()) keysrc += std::string("|") + o;
  char key[32] = {0};
  snprintf(key, sizeof key, "%016llx", (unsigned long long)fnv1a(keysrc, headers_hash(inc)));
  const std::string base = dir.empty() ? std::string() : dir + "/" + key;
  if (!base.empty()) {
    std::string bin, nm;
    if (read_file(base + ".cubin", &bin) && read_file(base + ".names", &nm) && !bin.empty()) {
      std::vector<std::string> lowered;
      std::istringstream in(nm);
      for (std::string line; std::getline(in, line);) lowered.push_back(line);
      if (lowered.size() == names.size()) {
        std::vector<char> cubin(bin.begin(), bin.end());
        if (finish_module(r, drv, cubin, lowered)) {
          r.from_cache = true;
          return r;
        }
        r = Module();  // unusable entry: compile afresh
      }
    }
  }
  if (!nv.ok) {
    r.why = nv.why;
    return r;
  }
  void* prog = nullptr;
  if (nv.create(&prog, src.c_str(), "df_generated.cu", 0, nullptr, nullptr) != 0) {
    r.why = "nvrtcCreateProgram failed";
    return r;
  }
  for (auto& s : names) nv.add_name(prog, s.c_str());
  const auto t0 = std::chrono::steady_clock::now();
  const int rc = nv.compile(prog, (int)(sizeof(opts) / sizeof(opts[0])), opts);
  r.compile_ms = (size_t)std::chrono::duration_cast<std::chrono::milliseconds>(std::chrono::steady_clock::now() - t0)
                     .count();
  if (rc != 0) {
    size_t n = 0;
    nv.log_size(prog, &n);
    std::string log(n, '\0');
    if (n) nv.log(prog, &log[0]);
    r.why = "NVRTC compilation failed: " + log.substr(0, 2000);
    nv.destroy(&prog);
    return r;
  }
  size_t nb = 0;
  nv.cubin_size(prog, &nb);
  std::vector<char> cubin(nb);
  nv.cubin(prog, cubin.data());
  std::vector<std::string> lowered;
  for (auto& s : names) {
    const char* l = nullptr;
    nv.lowered(prog, s.c_str(), &l);
    lowered.push_back(l ? std::string(l) : std::string());
  }
  nv.destroy(&prog);
  if (!base.empty()) {  // best effort: a failed write only costs the next process a compile
    std::string nm;
    for (auto& l : lowered) nm += l + "\n";
    if (write_file_atomic(base + ".cubin", std::string(cubin.begin(), cubin.end())))
      write_file_atomic(base + ".names", nm);
  }
  if (!finish_module(r, drv, cubin, lowered)) {
    r.cubin = cubin;
    r.lowered = lowered;
    r.retries = 3;
  }
  return r;
}

}  // namespace

int jit_thread_launch(df_mech* m, int threads, int bps, const IntegArgs& a, bool order, cudaStream_t st,
                      bool* launched) {
  *launched = false;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return DF_OK;
  // the variant that refines the ignition time has one block size
  int variant = a.t_ign ? kIgnVariant : 0;
  while (variant < kIgnVariant && kVariantThreads[variant] != threads) ++variant;
  if (!a.t_ign && variant == kIgnVariant) return DF_OK;  // no generated kernel for this block size
  threads = kVariantThreads[variant];
  Module* md = static_cast<Module*>(m->jit_module[dev][variant]);
  if (!md) {  // first launch on this device: generate, and compile unless cached
    const std::string src = jit_thread_source(m);
    std::lock_guard<std::mutex> lock(g_mu);
    const RelaxedCapture relaxed;
    auto key = std::make_pair(dev * kVariants + variant, src);
    auto it = g_modules.find(key);
    if (it == g_modules.end()) {
      it = g_modules.emplace(key, build_module(dev, m, src, variant)).first;
      const Systems sys = systems_of(m, reactions_of(m));
      it->second.per_thread = sys.per_thread() + Systems::exponents();
    } else if (it->second.retries > 0) {
      Module& r = it->second;
      r.retries = finish_module(r, driver(), r.cubin, r.lowered) ? 0 : r.retries - 1;
    }
    md = &it->second;
    if (md->retries == 0) {
      md->cubin = {};
      m->jit_module[dev][variant] = md;
    }
    m->jit_note = !md->ok          ? md->why
                  : md->from_cache ? std::string("generated kernel loaded from the on-disk cache")
                                   : "generated kernel compiled in " + std::to_string(md->compile_ms) + " ms";
  }
  if (!md->ok) return DF_OK;
  const CUfunction fk = md->fn;
  const Driver& drv = driver();
  const int per_thread = md->per_thread;
  IntegArgs args = a;
  // the mechanism if staging it leaves as many blocks on an SM as reading it
  // through L1, the per-thread workspace
  const size_t sm_staged = sizeof(double) * ((size_t)blob_smem_doubles(m->dims) + (size_t)per_thread * threads);
  const size_t sm_plain = sizeof(double) * (size_t)per_thread * threads;
  auto blocks_per_sm = [m](size_t b) {
    return b > m->max_smem_optin ? (size_t)0 : m->smem_per_sm / (b + m->smem_reserved_per_block);
  };
  args.stage_blob = blocks_per_sm(sm_staged) >= blocks_per_sm(sm_plain) ? 1 : 0;
  const size_t sm = args.stage_blob ? sm_staged : sm_plain;
  if (sm > m->max_smem_optin) return DF_OK;
  if (drv.set_attr(fk, CU_FUNC_ATTRIBUTE_MAX_DYNAMIC_SHARED_SIZE_BYTES, (int)sm) != CUDA_SUCCESS)
    return set_error(DF_ECUDA, "generated integrator: shared-memory attribute");
  int occ = 0;
  if (drv.occupancy(&occ, fk, threads, sm) != CUDA_SUCCESS || occ < 1)
    return set_error(DF_ECUDA, "generated integrator: occupancy query");
  const int per_sm = bps > 0 ? std::min(bps, occ) : occ;
  int64_t blocks = (int64_t)m->num_sms * per_sm;
  const int64_t need = (args.nwork + threads - 1) / threads;
  if (blocks > need) blocks = std::max<int64_t>(1, need);
  int rc = order_unless_alone(m, args, order, per_sm, threads / 32, 32, st);
  if (!rc) rc = cuda_check(cudaMemsetAsync(m->counters, 0, 4 * sizeof(unsigned long long), st), "reset work counter");
  if (rc) return rc;
  void* params[] = {&args};
  if (drv.launch(fk, (unsigned)blocks, 1, 1, (unsigned)threads, 1, 1, (unsigned)sm, (CUstream)st, params,
                 nullptr) != CUDA_SUCCESS)
    return set_error(DF_ECUDA, "generated integrator launch");
  *launched = true;
  m->jit_used = 1;
  return DF_OK;
}

}  // namespace df
