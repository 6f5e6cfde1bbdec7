// Source term and Jacobian of few cells, one cell per warp: the operations of
// eval_thread, spread over the lanes.  Each value is formed by one lane with the
// expressions of eval_thread, and every sum runs over the same terms in the same order,
// so a cell's bits do not depend on which of the two forms its batch takes:
//   species k       lane k: cp, h, g and C; its production rate and its row of J
//   reaction j      lane j mod 32: its rate and derivatives, through shared memory
//   temperature row lane c: its column c
// Where two products meet in a sum the text says which one is fused, here as there.
// What bounds it: latency, one warp's chains on an FP64 pipe (64 cycles per instruction
// whatever the number of active lanes).  9 species, 25 reactions, kernel and launch: source
// term 14.4 us up to four cells per SM (43 for a thread per cell), Jacobian 28.7 (154).
#pragma once
#include "chem_thread.cuh"

namespace df {

// the occurrences of species k among the reactions' entries, in eval_thread's order:
// occ[occ[k]] .. occ[occ[k + 1]] hold 8 j + a, entry a of reaction j (reactants 0-2,
// products 3-5)

// per-warp workspace (offsets in doubles)
struct LanesWS {
  int y, f, C, gRT, hRT, cpR, wdot, t, q, J, dT, d, dM, total;
};

__host__ __device__ inline LanesWS lanes_ws_layout(int N, int M, int n_eff, bool with_J) {
  const int n = N + 1;
  LanesWS w;
  int o = 0;
  w.y = o; o += n;
  w.f = o; o += n;
  w.C = o; o += N;
  w.gRT = o; o += N;
  w.hRT = o; o += N;
  w.cpR = o; o += N;
  w.wdot = o; o += N;
  w.t = o; o += 2 * N;
  w.q = o; o += M;
  w.J = w.dT = w.d = w.dM = o;
  if (with_J) {
    o += n * n;
    w.dT = o; o += M;
    w.d = o; o += 6 * M;
    w.dM = o; o += n_eff;
  }
  w.total = (o + 1) & ~1;
  return w;
}

// y at ws + L.y (T, Y) -> f at ws + L.f, J at ws + L.J; returns qdot in erg/(cm^3 s)
template <int NS, bool WITH_J>
__device__ __forceinline__ double eval_lanes(const MechView& mv, const int* occ, double pc, double* ws, const LanesWS& L) {
  constexpr int n = NS + 1;
  constexpr unsigned ALL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const double* y = ws + L.y;
  double* tmp = ws + L.t;
  SV C{ws + L.C, 1}, gRT{ws + L.gRT, 1}, hRT{ws + L.hRT, 1}, cpR{ws + L.cpR, 1}, wdot{ws + L.wdot, 1};
  const double T = y[0], invT = 1.0 / T;
  const bool species = lane < NS;
  const int k = species ? lane : 0;
  const double* a = mv.sp + SP_REC * k + 2;
  const double iW = mv.sp[SP_REC * k + 1];
  if (species) {
    const double cpk = a[0] + T * (a[1] + T * (a[2] + T * (a[3] + T * a[4])));
    cpR[k] = cpk;
    tmp[k] = y[1 + k] * cpk;
  }
  __syncwarp();
  // sum Y/W by the even lanes, cp by the odd ones
  const double* terms = (lane & 1) ? tmp : y + 1;
  double sum = 0.0;
#pragma unroll
  for (int l = 0; l < NS; ++l) sum += terms[l] * mv.sp[SP_REC * l + 1];
  const double sumYW = __shfl_sync(ALL, sum, 0);
  double cpm = __shfl_sync(ALL, sum, 1);
  const bool fixed = fixed_covers(mv, T) && rcp_in_range(sumYW) && rcp_in_range(pc);
  FixState fst;
  double lnT = 0.0;
  if (fixed) fst = fix_state(T, invT);
  else lnT = fast_log(T);
  cpm = cpm * RU;
  const double rho = pc * invT / (RU * sumYW);
  // three reciprocals as one
  const double rcp = 1.0 / (lane == 0 ? rho : lane == 1 ? cpm : sumYW);
  const double invrho = __shfl_sync(ALL, rcp, 0), invcp = __shfl_sync(ALL, rcp, 1), Wbar = __shfl_sync(ALL, rcp, 2);
  if (species) {
    const double* ah = mv.sp + SP_REC * k + SP_H;
    const double hk = a[0] + T * (ah[0] + T * (ah[1] + T * (ah[2] + T * ah[3]))) + a[5] * invT;
    hRT[k] = hk;
    if (fixed) {
      gRT[k] = __longlong_as_double(fix_gibbs(mv.fix + mv.fg + 7 * k, fst));
    } else {
      const double* as = mv.sp + SP_REC * k + SP_S;
      const double sk = a[0] * lnT + T * (a[1] + T * (as[0] + T * (as[1] + T * as[2]))) + a[6];
      gRT[k] = hk - sk;
    }
    C[k] = rho * y[1 + k] * iW;
  }
  __syncwarp();
  const double lnP0RT = LOG_PSTD_RU - lnT;
  for (int j = lane; j < mv.M; j += 32) {
    RateOut ro;
    if (fixed) rate_fixed<NS, WITH_J>(mv, j, mv.rx + RX_REC * j, NS, T, invT, fst, C, gRT, hRT, ro);
    else
      rate_one<NS, WITH_J>(mv, mv.rx + RX_REC * j, NS, T, lnT, invT, lnP0RT, C, gRT, hRT, ro);
    // no rate: zeros, which leave the sums as they are
    ws[L.q + j] = ro.active ? ro.q : 0.0;
    if (WITH_J) {
      double* d = ws + L.d + 6 * j;
      if (ro.active) {
        ws[L.dT + j] = ro.dqdT;
        d[0] = ro.fk * ro.cr[1] * ro.cr[2];
        d[1] = ro.fk * ro.cr[0] * ro.cr[2];
        d[2] = ro.fk * ro.cr[0] * ro.cr[1];
        d[3] = -(ro.rk * ro.cp[1] * ro.cp[2]);
        d[4] = -(ro.rk * ro.cp[0] * ro.cp[2]);
        d[5] = -(ro.rk * ro.cp[0] * ro.cp[1]);
        if ((ro.mt.flags & 3) != 0) ws[L.dM + ro.sl.eff] = ro.dqdM;
      } else {
        ws[L.dT + j] = 0.0;
        for (int i = 0; i < 6; ++i) d[i] = 0.0;
        const double* r = mv.rx + RX_REC * j;
        if ((load_meta(r).flags & 3) != 0) ws[L.dM + load_slots(r).eff] = 0.0;
      }
    }
  }
  __syncwarp();
  const int o0 = species ? occ[k] : 0, o1 = species ? occ[k + 1] : 0;
  double* row = ws + L.J + (1 + k) * n;
  if (WITH_J && species) {
#pragma unroll
    for (int c = 0; c < n; ++c) row[c] = 0.0;
  }
  double w = 0.0;
  for (int o = o0; o < o1; ++o) {
    const int e = occ[o], j = e >> 3;
    const bool isr = (e & 7) < 3;
    const double q = ws[L.q + j];
    w = isr ? w - q : w + q;
    if (WITH_J) {
      const double* r = mv.rx + RX_REC * j;
      const RxMeta mt = load_meta(r);
      const int nr = mt.nrnp & 15, np = mt.nrnp >> 4;
      const double sgn = isr ? -1.0 : 1.0;
      const double* d = ws + L.d + 6 * j;
      row[0] += sgn * ws[L.dT + j];
      row[1 + mt.reac[0]] += sgn * d[0];
      if (nr > 1) row[1 + mt.reac[1]] += sgn * d[1];
      if (nr > 2) row[1 + mt.reac[2]] += sgn * d[2];
      row[1 + mt.prod[0]] += sgn * d[3];
      if (np > 1) row[1 + mt.prod[1]] += sgn * d[4];
      if (np > 2) row[1 + mt.prod[2]] += sgn * d[5];
      if ((mt.flags & 3) != 0) {
        const int sl = load_slots(r).eff;
        const double* ef = mv.eff + NS * sl;
        const double cM = sgn * ws[L.dM + sl];
#pragma unroll
        for (int l = 0; l < NS; ++l) row[1 + l] += cM * ef[l];
      }
    }
  }
  if (species) wdot[k] = w;
  __syncwarp();
  double Hw = 0.0;
#pragma unroll
  for (int l = 0; l < NS; ++l) Hw += hRT[l] * wdot[l];
  Hw = Hw * (RU * T);
  const double fT = -(Hw * invrho * invcp);
  if (species) ws[L.f + 1 + k] = mv.sp[SP_REC * k] * w * invrho;
  if (lane == 0) ws[L.f] = fT;
  if (WITH_J) {
    if (species) {
      const double Wk = mv.sp[SP_REC * k];
      double s = 0.0;
#pragma unroll
      for (int l = 0; l < NS; ++l) s += row[1 + l] * C[l];
      const double aa = Wk * Wbar * invrho * (w - s);
#pragma unroll
      for (int i = 0; i < NS; ++i) row[1 + i] = (Wk * row[1 + i] + aa) * mv.sp[SP_REC * i + 1];
      row[0] = Wk * invrho * (row[0] + (w - s) * invT);
      tmp[k] = y[1 + k] * (a[1] + T * (2.0 * a[2] + T * (3.0 * a[3] + T * 4.0 * a[4])));
      tmp[NS + k] = cpR[k] * iW;
    }
    __syncwarp();
    // d cp/dT by the even lanes, sum of cp_k f_k by the odd ones
    double acc2 = 0.0;
#pragma unroll
    for (int l = 0; l < NS; ++l)
      acc2 += ((lane & 1) ? tmp[NS + l] : tmp[l]) * ((lane & 1) ? ws[L.f + 1 + l] : mv.sp[SP_REC * l + 1]);
    const double dcp = __shfl_sync(ALL, acc2, 0) * RU, cpf = __shfl_sync(ALL, acc2, 1);
    if (lane < n) {
      double acc = 0.0;
#pragma unroll
      for (int l = 0; l < NS; ++l) acc += hRT[l] * mv.sp[SP_REC * l + 1] * ws[L.J + (1 + l) * n + lane];
      acc = acc * (RU * T);
      double v;
      if (lane == 0) {
        v = fma(-invcp, fma(cpf, RU, acc), -(fT * dcp * invcp));
      } else {
        const double cpj = RU * cpR[lane - 1] * mv.sp[SP_REC * (lane - 1) + 1];
        v = fma(-(fT * cpj), invcp, -(invcp * acc));
      }
      ws[L.J + lane] = v;
    }
    __syncwarp();
  }
  return -Hw;
}

}  // namespace df
