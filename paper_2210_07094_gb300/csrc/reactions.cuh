// Host side: a mechanism's reactions as lists, the digits of the fixed-point rate
// arguments and the temperatures they cover (mech.cu writes them behind the blob,
// codegen.cu into the generated kernels).
#pragma once
#include <algorithm>
#include <cmath>
#include <vector>

#include "common.cuh"
#include "exp2fix.cuh"

namespace df {

inline RxMeta meta_of(const df_mech* m, int j) {
  RxMeta mt;
  memcpy(&mt, &m->blob_host[m->dims.off_rx + RX_REC * j + 3], 8);
  return mt;
}
inline RxSlots slots_of(const df_mech* m, int j) {
  RxSlots sl;
  memcpy(&sl, &m->blob_host[m->dims.off_rx + RX_REC * j + 4], 8);
  return sl;
}

struct Rx {
  std::vector<int> r, p;  // species entries
  std::vector<int> nu;    // net coefficients, by species
  std::vector<int> spc;   // species of the reaction
  int type = 0, eff = -1, troe = -1, dnu = 0;
  bool rev = false;
  double b = 0, E = 0;
};

inline std::vector<Rx> reactions_of(const df_mech* m) {
  std::vector<Rx> out(m->dims.M);
  for (int j = 0; j < m->dims.M; ++j) {
    Rx& x = out[j];
    const RxMeta mt = meta_of(m, j);
    const RxSlots sl = slots_of(m, j);
    for (int i = 0; i < (mt.nrnp & 15); ++i) x.r.push_back(mt.reac[i]);
    for (int i = 0; i < (mt.nrnp >> 4); ++i) x.p.push_back(mt.prod[i]);
    x.nu.assign(m->dims.N, 0);
    for (int k : x.r) x.nu[k] -= 1;
    for (int k : x.p) x.nu[k] += 1;
    for (const auto* side : {&x.r, &x.p})
      for (int k : *side)
        if (std::find(x.spc.begin(), x.spc.end(), k) == x.spc.end()) x.spc.push_back(k);
    x.type = mt.flags & 3;
    x.rev = (mt.flags & 4) != 0;
    x.eff = sl.eff;
    x.troe = sl.troe;
    x.dnu = (int)x.p.size() - (int)x.r.size();
    x.b = m->blob_host[m->dims.off_rx + RX_REC * j + 1];
    x.E = m->blob_host[m->dims.off_rx + RX_REC * j + 2];
  }
  return out;
}

// |c| 2^s, or |c| log2(e) 2^s, as a 64-bit integer and the left shift its use
// still needs (0 unless the value is too large for 64 bits).  Integer
// arithmetic only: the same digits on every host.
inline void fixed_literal(double c, bool log2e, int s, uint64_t* lit, int* shift) {
  *lit = 0;
  *shift = 0;
  if (c == 0.0) return;
  int e;
  const uint64_t m = (uint64_t)std::ldexp(std::frexp(std::fabs(c), &e), 53);  // |c| = m 2^(e - 53)
  const unsigned __int128 p = log2e ? (unsigned __int128)m * EXP2FIX_LOG2E_HALF : (unsigned __int128)m << 63;
  int bits = 64;
  while (bits < 128 && (p >> bits) != 0) ++bits;
  const int r0 = 116 - e - s;  // |c| (log2 e) 2^s = p 2^-r0
  int r = std::max(r0, bits - 64);
  if (r > 126) return;
  unsigned __int128 v = (p + ((unsigned __int128)1 << (r - 1))) >> r;
  if ((v >> 64) != 0) {
    ++r;
    v = (p + ((unsigned __int128)1 << (r - 1))) >> r;
  }
  *lit = (uint64_t)v;
  *shift = r - r0;
}

// the temperatures the fixed-point evaluation covers: from the lowest one at
// which every exponent, with any ln A of lnA_fits_fixed, stays below 1000 octaves
// and each of its parts within them (sampled every 2% and with 5% to spare); 0 if
// there is none.  saturating: the exponent of a reverse constant may fall below
// -1000 octaves (add_exponents).
inline double fixed_T_low(const df_mech* m, const std::vector<Rx>& rx, bool saturating) {
  const double L2E = 1.4426950408889634;
  auto sp = [&](int k, int i) { return m->blob_host[m->dims.off_sp + SP_REC * k + i]; };
  for (double lo : {100.0, 150.0, 200.0, 250.0, 300.0, 400.0}) {
    double worst = 0.0, least = 0.0;
    for (double T = lo; T < FIX_T_HIGH * 1.02; T *= 1.02) {
      std::vector<double> g(m->dims.N), h(m->dims.N);
      for (int k = 0; k < m->dims.N; ++k) {
        h[k] = sp(k, 2) + T * (sp(k, SP_H) + T * (sp(k, SP_H + 1) + T * (sp(k, SP_H + 2) + T * sp(k, SP_H + 3)))) +
               sp(k, 7) / T;
        worst = std::max(worst, std::fabs(h[k]));
        g[k] = L2E * ((sp(k, 2) - sp(k, 8)) - sp(k, 2) * std::log(T) -
                      T * (sp(k, 3) / 2 + T * (sp(k, 4) / 6 + T * (sp(k, 5) / 12 + T * sp(k, 6) / 20))) + sp(k, 7) / T);
      }
      for (const Rx& x : rx) {
        worst = std::max(worst, std::fabs(x.b) + std::fabs(x.E) / T);
        const double kf = 150.0 + L2E * std::fabs(x.b * std::log(T) - x.E / T);
        double sg = -x.dnu * L2E * (LOG_PSTD_RU - std::log(T)), sh = -x.dnu;
        for (int k : x.spc) {
          sg += x.nu[k] * g[k];
          sh += x.nu[k] * h[k];
        }
        worst = std::max({worst, kf + std::max(sg, 0.0), std::fabs(sg), std::fabs(sh)});
        least = std::max(least, kf - sg);
        if (x.type == 2) {
          const double* tr = &m->blob_host[m->dims.off_tr + TR_REC * x.troe];
          // the centring must be a positive number for its logarithm
          const double Fc = (1.0 - tr[3]) * std::exp(-T * tr[4]) + tr[3] * std::exp(-T * tr[5]) + std::exp(-tr[6] / T);
          if (!(Fc > 1e-60 && Fc < 1e60)) worst = INFINITY;
          const double d = L2E * std::fabs(tr[0] + (tr[1] - x.b) * std::log(T) - (tr[2] - x.E) / T);
          if (tr[0] != -INFINITY) worst = std::max({worst, d, kf + d, std::fabs(sg)});  // else it has no rate
        }
      }
    }
    // false for NaN and infinity
    if (worst * 1.05 <= 1000.0 && (saturating || least * 1.05 <= 1000.0)) return lo;
  }
  return 0.0;
}

}  // namespace df
