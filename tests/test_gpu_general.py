"""The generated integrator on cells of which the fixed-point evaluation covers none or
only some states (its general FP64 evaluation): a ln A beyond the fixed-point words,
temperatures below and above the covered ones, against the mechanism-independent
kernel, within test_gpu_jit's bounds."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2210_07094_gb300 as df  # noqa: E402
import test_gpu_jit as jit  # noqa: E402
from paper_2210_07094_gb300 import synth  # noqa: E402


@pytest.mark.parametrize("kind", ["ln_a", "cold", "hot"])
def test_general_evaluation(kind):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    mech = synth.h2_air_mechanism()
    m = df.Mechanism(mech)
    f = synth.field(1, mech, 600, seed=15)
    T0, p, Y0 = jit._dev(f)
    dt = f["dt"]
    r = np.random.default_rng(16)
    if kind == "ln_a":
        lnA = torch.tensor([np.log(x["A"]) for x in mech["reactions"]], dtype=torch.float64, device="cuda")
        lnA[7] = -105.0
        m.set_lnA(lnA)
    else:  # burnt-gas radicals, which recombine at any temperature; cells on both sides of the line
        Y0 = torch.tensor(10.0 ** r.uniform(-4.0, 0.0, (9, 600)), device="cuda")
        Y0 /= Y0.sum(0)
        lo, hi, dt = (60.0, 160.0, 1e-8) if kind == "cold" else (7950.0, 8200.0, 1e-9)
        T0 = torch.tensor(r.uniform(lo, hi, 600), device="cuda")
    ref, used, _ = jit._run(m, T0, p, Y0, dt, 32, 1)
    assert not used and (ref[2] == 0).float().mean() > 0.9
    out, used, detail = jit._run(m, T0, p, Y0, dt, 32, 0)
    assert used, detail
    print(kind, (ref[0] - T0).abs().max().item(), jit._close(ref, out))
    assert (ref[0] - T0).abs().max() > 1e-3  # the reactions do something
