"""GenEval::run of a generated kernel on the states that the fixed-point evaluation
leaves to the general FP64 one: below and above its temperatures, with a ln A beyond its
words, with mass fractions of any size.  The host build of test_gen_fixed_host with a
driver of its own; the reference is gen_eval, which that test compares over the
range, its Jacobian reduced to the systems' rows and columns here."""
import pytest

import test_gen_fixed_host as host

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
  std::mt19937_64 r(3);
  auto U = [&] { return (r() >> 11) * 0x1p-53; };
  auto sv = [](double* p) { return SVT<double, 1>{p, 1}; };
  auto* fix = reinterpret_cast<long long*>(blob.data() + d.off_fix());
  const long long flag = fix[d.M];
  int seen[4] = {}, covered[4] = {};
  double wf = 0;
  for (int t = 0; t < 4000; ++t) {
    const int kind = t & 3;
    double y[n], y2[n], f[n], g[n], fe[n], f2[n], J[n * n], sM[n], ex[128], W[GenEval::kWords], W0[GenEval::kWords], s = 0;
    y[0] = kind == 0 ? 40.0 + 260.0 * U() : kind == 1 ? 7900.0 + 3000.0 * U() : 300.0 + 3000.0 * U();
    for (int k = 0; k < N; ++k) s += y[1 + k] = pow(10.0, -9.0 * U());
    if (kind == 3) s *= pow(10.0, 64.0 * (U() - 0.5));
    for (int k = 0; k < N; ++k) y[1 + k] /= s;
    const double pc = 1.01325e6 * pow(10.0, 2.0 * U() - 0.5);
    fix[d.M] = kind == 2 ? 0 : flag;
    const MechView mv = make_view(blob.data(), d, blob.data());
    const bool in = gen_fixed<true, 1>(mv, pc, y, f, sv(W), sv(ex));
    GenEval::run<true, 1>(mv, pc, y, f, sv(W), sv(ex));
    GenEval::run<false, 1>(mv, pc, y, g, sv(W0), sv(ex));
    gen_eval<true, 1>(mv, pc, y, fe, sv(J), sv(sM));
    bool fin = true;
    for (double v : fe) fin = fin && isfinite(v);
    for (double v : J) fin = fin && isfinite(v);
    covered[kind] += in;
    seen[kind] += fin && !in;
    if (!in) {  // the same numbers: NaN and infinity where the reference has them
      auto same = [](double a, double b) { return a == b || (a != a && b != b); };
      for (int i = 0; i < n; ++i)
        if (!same(f[i], fe[i])) return 3;
      for (int a = 0; a < NA; ++a) {
        const int ra = GenEval::act(a);
        if (!same(g[ra], fe[ra])) return 4;
        for (int b = 0; b < NA; ++b) {
          double v = J[ra * n + GenEval::act(b)];
          for (int e = 0; e < GenEval::kNE; ++e) v += GenEval::beta(e, b) * J[ra * n + GenEval::elim(e)];
          if (!same(W[a * NA + b], -v)) return 5;
        }
      }
    } else if (kind == 3 && fin) {  // the temperature's rate divides by the heat capacity
      for (int i = 0; i < n; ++i) y2[i] = i ? y[i] : y[i] * (1 + 4e-16);
      gen_eval<true, 1>(mv, pc, y2, f2, sv(J), sv(sM));
      double cp = 0, f0 = 0;
      for (int k = 0; k < N; ++k) {
        const double* c = mv.sp + SP_REC * k + 2;
        const double T = y[0], iW = mv.sp[SP_REC * k + 1];
        cp += y[1 + k] * iW * (c[0] + T * (c[1] + T * (c[2] + T * (c[3] + T * c[4]))));
        f0 += fabs(T * iW * fe[1 + k] * (c[0] + T * (c[1] / 2 + T * (c[2] / 3 + T * (c[3] / 4 + T * c[4] / 5))) + c[5] / T));
      }
      const double e = fabs(f[0] - fe[0]) / (100 * fabs(f2[0] - fe[0]) + 1e-11 * f0 / fabs(cp) + 1e-280);
      if (!(e <= wf)) wf = e;
    }
  }
  printf("general %d %d %d %d covered %d %d %d %d f %g\n", seen[0], seen[1], seen[2], seen[3], covered[0], covered[1],
         covered[2], covered[3], wf);
  // each kind reaches the general evaluation with finite rates, mass fractions of most sizes do not need it
  return seen[0] >= 100 && seen[1] >= 500 && seen[2] >= 900 && seen[3] >= 10 && covered[2] == 0 && covered[3] >= 800 && wf <= 1 ? 0 : 1;
}
"""


@pytest.mark.parametrize("name", list(host.MECHS))
def test_states_outside_the_fixed_point_range(name, tmp_path, monkeypatch):
    """General evaluation: equal numbers.  Covered: the bounds of test_gen_fixed_host."""
    monkeypatch.setattr(host, "DRIVER", DRIVER)
    host.test_fixed_point_evaluation_matches_fp64(name, tmp_path)
