"""The adjoint's one-pass second-derivative terms (second_order) on the host, for
all reaction forms: against central differences of the transposed Jacobian products
(eval_vjp) along each stage vector, summed over the stages."""
import shutil
import subprocess

import pytest

from paper_2210_07094_gb300 import synth
from test_gen_fixed_host import BUILD, CSRC, DUMP, MECHS, NVCC, STUB

DRIVER = r"""
#include "stub.h"
#include "gen.cu"
using namespace df;
int main() {
  constexpr int N = GenEval::kN, n = N + 1, NS = 6, MX = 64;
  FILE* fp = fopen("blob.bin", "rb");
  MechDims d;
  if (fread(&d, sizeof d, 1, fp) != 1) return 2;
  std::vector<double> blob(d.allocated());
  if (fread(blob.data(), 8, blob.size(), fp) != blob.size() || d.M > MX) return 2;
  MechView mv = make_view(blob.data(), d, blob.data());
  mv.T_low = INFINITY;  // FP64 rates, the smoother function to difference
  std::mt19937_64 r(1);
  auto U = [&] { return (r() >> 11) * 0x1p-53; };
  double worst = 0;
  for (int t = 0; t < 200; ++t) {
    double y[n], K[NS * n], R[NS * n], b[n] = {}, th[MX] = {}, s = 0, vec[7][N];
    y[0] = 500.0 + 2300.0 * U();
    for (int k = 0; k < N; ++k) s += y[1 + k] = pow(10.0, -3.0 * U());
    for (int k = 0; k < N; ++k) y[1 + k] /= s;
    for (int i = 0; i < NS * n; ++i) {
      K[i] = (U() - 0.5) * y[i % n];
      R[i] = (U() - 0.5) * (i % n ? 1.0 : 1e-3);
    }
    const double pc = 1.01325e6 * pow(10.0, 2.0 * U() - 0.5);
    SV V[7];
    for (int i = 0; i < 7; ++i) V[i] = SV{vec[i], 1};
    second_order<N>(mv, pc, y, NS, SV{K, 1}, SV{R, 1}, b, V[0], V[1], V[2], V[3], V[4], V[5], SV{th, 1});
    // sum over the stages of J(y + e K)^T r and of r . df/d ln A there
    double sc[n + MX] = {};
    auto products = [&](double e, double* out) {
      for (int i = 0; i < n + MX; ++i) out[i] = 0.0;
      for (int q = 0; q < NS; ++q) {
        double z[n], rr[n], bb[n], f[n], u[N], t1[MX] = {};
        for (int i = 0; i < n; ++i) z[i] = y[i] + e * K[q * n + i];
        for (int i = 0; i < n; ++i) rr[i] = R[q * n + i];
        ThetaHook hk{1, 0.0, SV{t1, 1}, SV{u, 1}};
        eval_vjp<N>(mv, pc, z, rr, bb, f, V[0], V[1], V[2], V[3], V[4], V[5], V[6], &hk);
        for (int i = 0; i < n + d.M; ++i) {
          const double x = i < n ? bb[i] : t1[i - n];
          out[i] += x;
          sc[i] = fmax(sc[i], fabs(x));
        }
      }
    };
    const double e = 1e-3;
    double p[4][n + MX];
    products(e, p[0]);
    products(-e, p[1]);
    products(2 * e, p[2]);
    products(-2 * e, p[3]);
    for (int i = 0; i < n + d.M; ++i) {
      const double D1 = (p[0][i] - p[1][i]) / (2 * e), D2 = (p[2][i] - p[3][i]) / (4 * e);
      const double got = i < n ? b[i] : th[i - n];
      const double w = fabs(got - (4 * D1 - D2) / 3) / (0.01 * fabs(D2 - D1) + 1e-9 * sc[i] + 1e-290);
      if (!(w <= worst)) worst = w;
    }
  }
  printf("worst %g\n", worst);
  return worst <= 1 ? 0 : 1;
}
"""


@pytest.mark.parametrize("name", ["h2_air", "isomer_three_body", "irreversible", "forms"])
def test_second_order_matches_differences(name, tmp_path):
    """Central differences with steps e = 1e-3 and 2e of the stage vector, extrapolated:
    what is left of the truncation is below a hundredth of their difference, and the
    rounding is the products' (1e-13 of their largest) over e, with a factor of ten."""
    if not shutil.which(NVCC) or not shutil.which("g++"):
        pytest.skip("no nvcc or g++")
    inc = tmp_path / "inc"
    shutil.copytree(CSRC, inc, ignore=lambda d, fs: [f for f in fs if not f.endswith((".cuh", ".inc"))])
    synth.write_json(MECHS[name](), str(tmp_path / "mech.json"))
    (tmp_path / "dump.cu").write_text(DUMP)
    run = lambda cmd: subprocess.run(cmd, cwd=tmp_path, capture_output=True, text=True)  # noqa: E731
    r = run([NVCC, "-std=c++17", "-I", CSRC, "-o", "dump", "dump.cu", "-L", BUILD, "-ldfchem", "-Xlinker", "-rpath=" + BUILD])
    assert r.returncode == 0, r.stderr[-2000:]
    assert run(["./dump", "mech.json"]).returncode == 0
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
