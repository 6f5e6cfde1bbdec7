"""The generated fixed-point evaluation (gen_fixed) and the mechanism-independent one
(eval_thread with rate_fixed) against the generated FP64 one (gen_eval) on the host: the same source text compiled by g++ with the device
intrinsics it uses written out, so that f and every Jacobian entry are compared
for all reaction forms without a GPU."""
import os
import shutil
import subprocess

import pytest

from paper_2210_07094_gb300 import synth

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2210_07094_gb300", "csrc")
BUILD = os.path.join(ROOT, "paper_2210_07094_gb300", "_build")
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"

STUB = r"""
#pragma once
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <random>
#include <vector>
using std::fabs; using std::fmax; using std::fmin; using std::isfinite;
#define __CUDACC__
#define __CUDACC_RTC__
#define __device__
#define __host__
#define __global__
#define __constant__
#define __shared__
#define __forceinline__ inline
#define __noinline__
#define __launch_bounds__(...)
#define __align__(x)
struct D3 { int x, y, z; };
static D3 threadIdx, blockIdx, blockDim, gridDim;
static inline uint32_t __umulhi(uint32_t a, uint32_t b) { return (uint32_t)(((uint64_t)a * b) >> 32); }
static inline int __clz(unsigned x) { return x ? __builtin_clz(x) : 32; }
static inline int __clzll(long long x) { return x ? __builtin_clzll(x) : 64; }
template <class T> T min(T a, T b) { return a < b ? a : b; }
template <class T> T max(T a, T b) { return a > b ? a : b; }
static inline uint64_t bits_of(double x) { uint64_t u; memcpy(&u, &x, 8); return u; }
static inline double of_bits(uint64_t u) { double x; memcpy(&x, &u, 8); return x; }
static inline int __double2hiint(double x) { return (int)(bits_of(x) >> 32); }
static inline int __double2loint(double x) { return (int)bits_of(x); }
static inline double __hiloint2double(int h, int l) { return of_bits((uint64_t)(uint32_t)h << 32 | (uint32_t)l); }
static inline double __longlong_as_double(long long u) { return of_bits(u); }
static inline long long __double_as_longlong(double x) { return bits_of(x); }
static inline void rcp_bits(uint32_t& r, uint32_t a) { float f; memcpy(&f, &a, 4); f = 1.0f / f; memcpy(&r, &f, 4); }
template <class T> T __ldg(const T* p) { return *p; }
template <class A, class B> unsigned long long atomicAdd(A*, B) { return 0; }
static inline unsigned __ballot_sync(unsigned, bool) { return 0; }
static inline int __ffs(unsigned) { return 0; }
static inline int __popc(unsigned) { return 0; }
template <class T> T __shfl_sync(unsigned, T v, int) { return v; }
template <class T> T __shfl_down_sync(unsigned, T v, int) { return v; }
static inline void __syncthreads() {}
static inline double __dsub_rn(double a, double b) { return a - b; }
"""

DRIVER = r"""
#include "stub.h"
#include "gen.cu"
using namespace df;
int main() {
  constexpr int N = GenEval::kN, n = N + 1, NA = GenEval::kNA;
  FILE* fp = fopen("blob.bin", "rb");
  MechDims d;
  if (fread(&d, sizeof d, 1, fp) != 1) return 2;
  std::vector<double> blob(d.allocated());
  if (fread(blob.data(), 8, blob.size(), fp) != blob.size()) return 2;
  MechView mv = make_view(blob.data(), d, blob.data());
  std::mt19937_64 r(1);
  auto U = [&] { return (r() >> 11) * 0x1p-53; };
  int inside = 0;
  double wf = 0, wj = 0, wp = 0, bf = 0, bj = 0;
  for (int t = 0; t < 2000; ++t) {
    double y[n], y2[n], f[n], fe[n], f2[n], fp_[n], W[GenEval::kWords], W0[GenEval::kWords], ex[128], J[n * n], J2[n * n], sM[n], s = 0;
    y[0] = t % 50 == 0 ? 30.0 + 12000.0 * U() : 240.0 + 3000.0 * U();
    for (int k = 0; k < N; ++k) s += y[1 + k] = pow(10.0, -9.0 * U()) * (U() < 0.05 ? -1e-6 : 1.0);
    for (int k = 0; k < N; ++k) y[1 + k] /= s;
    const double pc = 1.01325e6 * pow(10.0, 2.0 * U() - 0.5);
    SVT<double, 1> E{ex, 1};
    for (double& v : W) v = NAN;
    for (double& v : W0) v = NAN;
    const bool in = gen_fixed<true, 1>(mv, pc, y, f, SVT<double, 1>{W, 1}, E);
    if (in != gen_fixed<false, 1>(mv, pc, y, fp_, SVT<double, 1>{W0, 1}, E)) return 3;
    if (!in) {
      for (double v : W) if (v == v) return 4;  // nothing may be written
      continue;
    }
    ++inside;
    for (int i = 0; i < n; ++i) y2[i] = y[i];
    y2[0] *= 1 + 4e-16;
    SVT<double, 1> S{sM, 1};
    gen_eval<true, 1>(mv, pc, y, fe, SVT<double, 1>{J, 1}, S);
    gen_eval<true, 1>(mv, pc, y2, f2, SVT<double, 1>{J2, 1}, S);
    double nf = 1e-300;
    for (int i = 1; i < n; ++i) nf = fmax(nf, fabs(fe[i]));
    // the temperature's rate sums h_k times the species' rates: its terms
    double f0 = 1e-300, cp0 = 0;
    for (int k = 0; k < N; ++k) {
      const double* c = mv.sp + SP_REC * k + 2;
      const double T = y[0], iW = mv.sp[SP_REC * k + 1];
      cp0 += y[1 + k] * iW * (c[0] + T * (c[1] + T * (c[2] + T * (c[3] + T * c[4]))));
      f0 += fabs(T * iW * fe[1 + k] * (c[0] + T * (c[1] / 2 + T * (c[2] / 3 + T * (c[3] / 4 + T * c[4] / 5))) + c[5] / T));
    }
    f0 /= fabs(cp0);
    for (int i = 0; i < n; ++i) {
      const double tol = 100 * fabs(f2[i] - fe[i]) + 1e-11 * (i ? nf : f0) + 1e-280;
      wf = fmax(wf, fabs(f[i] - fe[i]) / tol);
      for (int a = 0; a < NA; ++a)  // without J only the systems' entries
        if (GenEval::act(a) == i) wp = fmax(wp, fabs(f[i] - fp_[i]) / tol);
    }
    // the mechanism-independent evaluation, which reads the same arguments from the blob
    // against itself in FP64 (no temperature covered)
    double fb[n], fs[n], fq[n], v5[5][N], Jb[n * n], Js[n * n], Jq[n * n], cf[n] = {}, cJ[n * n] = {};
    MechView mvs = mv;
    mvs.T_low = INFINITY;
    auto sv = [](double* p) { return SVT<double, 1>{p, 1}; };
    auto blob_eval = [&](const MechView& v, const double(&z)[n], double(&ff)[n], double* JJ) {
      eval_thread<N, true, double, false, 1>(v, pc, z, ff, sv(v5[0]), sv(v5[1]), sv(v5[2]), sv(v5[3]), sv(v5[4]), sv(JJ));
    };
    blob_eval(mv, y, fb, Jb);
    blob_eval(mvs, y, fs, Js);
    for (int q = 0; q < n; ++q) {  // the change with each entry of the state (1 + 4e-16)
      double z[n];
      for (int i = 0; i < n; ++i) z[i] = y[i] * (i == q ? 1 + 4e-16 : 1);
      blob_eval(mvs, z, fq, Jq);
      for (int i = 0; i < n; ++i) cf[i] = fmax(cf[i], fabs(fq[i] - fs[i]));
      for (int i = 0; i < n * n; ++i) cJ[i] = fmax(cJ[i], fabs(Jq[i] - Js[i]));
    }
    for (int i = 0; i < n; ++i)
      bf = fmax(bf, fabs(fb[i] - fs[i]) / (100 * cf[i] + 1e-11 * (i ? nf : f0) + 1e-280));
    // the columns over the kept species: beta times the eliminated ones' added
    auto red = [&](const double* A, int ra, int b) {
      double v = A[ra + GenEval::act(b)];
      for (int e = 0; e < GenEval::kNE; ++e) v += GenEval::beta(e, b) * A[ra + GenEval::elim(e)];
      return v;
    };
    for (int a = 0; a < NA; ++a) {
      double nr = 1e-300;
      const int ra = GenEval::act(a) * n;
      for (int j = 0; j < n; ++j) nr = fmax(nr, fabs(J[ra + j]));
      if (ra == 0) {  // the temperature row sums h_k times the species rows: its terms
        const double T = y[0];
        double cp = 0;
        for (int k = 0; k < N; ++k) {
          const double* c = mv.sp + SP_REC * k + 2;
          cp += y[1 + k] * mv.sp[SP_REC * k + 1] * (c[0] + T * (c[1] + T * (c[2] + T * (c[3] + T * c[4]))));
        }
        for (int j = 0; j < n; ++j) {
          double s = 0;
          for (int k = 0; k < N; ++k) {
            const double* c = mv.sp + SP_REC * k + 2;
            const double h = c[0] + T * (c[1] / 2 + T * (c[2] / 3 + T * (c[3] / 4 + T * c[4] / 5))) + c[5] / T;
            s += fabs(T * h * mv.sp[SP_REC * k + 1] * J[(1 + k) * n + j]);
          }
          nr = fmax(nr, s / fabs(cp));
        }
      }
      for (int b = 0; b < NA; ++b) {
        const int id = ra + GenEval::act(b);
        const double d = fabs(Jb[id] - Js[id]) / (100 * cJ[id] + 1e-11 * nr);
        if (!(d <= bj)) bj = d;
        const double j = red(J, ra, b), e = fabs(W[a * NA + b] + j) / (100 * fabs(red(J2, ra, b) - j) + 1e-11 * nr);
        if (!(e <= wj)) wj = e;
      }
    }
    auto row_max = [&](int i) {
      double v = 0;
      for (int j = 0; j < n; ++j) v = fmax(v, fabs(J[i * n + j]));
      return v;
    };
    for (int i = 0; i < n; ++i) {  // the other rows are zero or follow from the systems'
      int e = 0, act = 0;
      for (int a = 0; a < NA; ++a) act += GenEval::act(a) == i;
      while (e < GenEval::kNE && GenEval::elim(e) != i) ++e;
      if (act + (e < GenEval::kNE) > 1) return 5;
      for (int j = -1; j < n && !act; ++j) {
        double v = j < 0 ? fe[i] : J[i * n + j], terms = j < 0 ? nf : row_max(i);
        for (int a = 0; a < NA && e < GenEval::kNE; ++a) {
          const int ra = GenEval::act(a);
          const double t = GenEval::beta(e, a) * (j < 0 ? fe[ra] : J[ra * n + j]);
          v -= t;
          terms += fabs(GenEval::beta(e, a)) * (j < 0 ? nf : row_max(ra));
        }
        if (!(fabs(v) <= 1e-11 * terms)) return 6;
        if (e == GenEval::kNE && f[i] != 0.0) return 7;
      }
    }
  }
  printf("inside %d f %g J %g plain %g blob f %g J %g\n", inside, wf, wj, wp, bf, bj);
  return inside >= 1000 && wf <= 1 && wj <= 1 && wp <= 1 && bf <= 1 && bj <= 1 && mv.T_low < 500 ? 0 : 1;
}
"""

DUMP = r"""
#include "common.cuh"
int main(int, char** v) {
  df_mech* m = new df_mech();
  if (df::parse_mechanism(v[1], m)) return 1;
  FILE* f = fopen("blob.bin", "wb");
  fwrite(&m->dims, sizeof(m->dims), 1, f);
  fwrite(m->blob_host.data(), 8, m->blob_host.size(), f);
  fclose(f);
  f = fopen("gen.cu", "w");
  const std::string s = df::jit_thread_source(m);
  fwrite(s.data(), 1, s.size(), f);
  return fclose(f);
}
"""


def _forms():
    """Every reaction form: one to three entries a side in all patterns of equal
    species, species on both sides, an inert catalyst, irreversible reactions,
    third bodies and falloff with efficiencies for reacting and inert species,
    full NASA-7 polynomials."""
    names = ["A", "B", "C", "D", "E", "X"]
    sp = [{"name": s, "composition": {"X": 1}, "W": 10.0 + 7.0 * i, "T_range": [300.0, 3000.0],
           "nasa7": [2.5 + 0.3 * i, 1e-3 * (i - 2), -2e-7 * (i - 3), 3e-11 * (i + 1), -1e-15 * i, -900.0 * i * i + 2000.0,
                     3.0 - i]} for i, s in enumerate(names)]
    sides = [{"A": 1}, {"A": 2}, {"B": 3}, {"A": 1, "B": 1}, {"A": 1, "B": 2}, {"A": 2, "C": 1}, {"B": 1, "C": 1, "D": 1},
             {"A": 1, "X": 1}, {"D": 1, "X": 2}, {"E": 1}, {"C": 2}]
    rx = []
    for i, a in enumerate(sides):
        b = sides[(3 * i + 4) % len(sides)]
        if "X" in a or "X" in b:  # X is inert: the same count on both sides
            a = {k: v for k, v in a.items() if k != "X"}
            b = {k: v for k, v in b.items() if k != "X"}
            if sum(a.values()) < 3 and sum(b.values()) < 3:
                a, b = {**a, "X": 1}, {**b, "X": 1}
        kind = ["elementary", "three-body", "elementary", "falloff-troe"][i % 4]
        r = {"reactants": a, "products": b, "type": kind, "reversible": i % 5 != 2, "A": 10.0 ** (4 + i), "b": 0.4 * (i - 5),
             "Ea": 15.0 * i - 20.0, "equation": ""}
        if kind != "elementary":
            r["efficiencies"] = {"A": 2.5, "X": 0.4, "E": 0.0}
        if kind == "falloff-troe":
            r["low"] = {"A": 10.0 ** (9 + i), "b": -0.7, "Ea": 10.0}
            r["troe"] = {"alpha": 0.6, "T3": 90.0, "T1": 1700.0, "T2": 4000.0}
        rx.append(r)
    return {"name": "forms", "elements": ["X"], "units": {"A": "cm, mol, s", "Ea": "kJ/mol", "T": "K"}, "species": sp,
            "reactions": rx}


MECHS = {"h2_air": synth.h2_air_mechanism,
         "chon_14": lambda: synth.hydrocarbon_mechanism(n_species=12, M=40, n_tb=4, n_troe=2),
         "isomer_three_body": lambda: synth.isomer_mechanism(kind="three-body", A=3e10, eff={"D": 2.5}),
         "irreversible": synth.autocatalytic_mechanism, "forms": _forms}


@pytest.mark.parametrize("name", list(MECHS))
def test_fixed_point_evaluation_matches_fp64(name, tmp_path):
    """The FP64 evaluation rounds its exponents (|ln k| up to several hundred) to
    1e-13: entries agree within that of the sum of their terms, of which a
    hundred times the entry's own change with T (1 + 4e-16), plus 1e-11 of the
    row (for the temperature row: of the h_k-weighted terms it sums), is a bound."""
    if not os.path.exists(NVCC) or not shutil.which("g++"):
        pytest.skip("no nvcc or g++")
    inc = tmp_path / "inc"
    shutil.copytree(CSRC, inc, ignore=lambda d, fs: [f for f in fs if not f.endswith((".cuh", ".inc"))])
    synth.write_json(MECHS[name](), str(tmp_path / "mech.json"))
    (tmp_path / "dump.cu").write_text(DUMP)
    run = lambda cmd: subprocess.run(cmd, cwd=tmp_path, capture_output=True, text=True)  # noqa: E731
    r = run([NVCC, "-std=c++17", "-I", CSRC, "-o", "dump", "dump.cu", "-L", BUILD, "-ldfchem", "-Xlinker", "-rpath=" + BUILD])
    assert r.returncode == 0, r.stderr[-2000:]
    assert run(["./dump", "mech.json"]).returncode == 0
    src = (tmp_path / "gen.cu").read_text()
    assert "gen_fixed<" in src
    # the text as it is, but for the PTX reciprocals and the dynamic shared memory
    dev = (inc / "dev_common.cuh").read_text()
    for a, b in (('asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r0f) : "f"((float)a));', "r0f = 1.0f / (float)a;"),
                 ('asm("rcp.approx.ftz.f32 %0, %1;" : "=r"(r) : "r"(((hi << 3) - 0xc0000000u) | sign));',
                  "rcp_bits(r, ((hi << 3) - 0xc0000000u) | sign);"),
                 ("typedef unsigned char uint8_t;\ntypedef int int32_t;\ntypedef unsigned int uint32_t;\n"
                  "typedef long long int64_t;\ntypedef unsigned long long uint64_t;\n", "")):
        assert a in dev
        dev = dev.replace(a, b)
    (inc / "dev_common.cuh").write_text(dev)
    k = (inc / "integrate_thread.cuh").read_text()
    (inc / "integrate_thread.cuh").write_text(k.replace("extern __shared__ double smem[];", "double smem[1];"))
    (tmp_path / "stub.h").write_text(STUB)
    (tmp_path / "driver.cpp").write_text(DRIVER)
    r = run(["g++", "-std=c++17", "-O1", "-w", "-I", str(inc), "-I", ".", "-o", "driver", "driver.cpp"])
    assert r.returncode == 0, r.stderr[-3000:]
    r = run(["./driver"])
    print(r.stdout)
    assert r.returncode == 0, (r.returncode, r.stdout)
