"""The warp path at the edges of its workspace layout and of its solves: fewer
and more reactions than the stage vectors' and the matrix's storage hold, orders
around 32 and 64, against the oracle; and a cell's result does not depend on how many
share its block."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2210_07094_gb300 as df  # noqa: E402
from oracle.oracle import Mech  # noqa: E402
from oracle.parity import check_integrator  # noqa: E402
from paper_2210_07094_gb300 import synth  # noqa: E402

DEV = "cuda:0"


def _dev(f):
    return (torch.tensor(f["T"], device=DEV), torch.tensor(f["p"], device=DEV),
            torch.tensor(np.ascontiguousarray(f["Y"]), device=DEV))


def _warp():
    o = df.default_opts()
    o.path = 2
    return o


MECHS = {  # order n, reactions M: the rate factors fit the stage vectors for M <= 6n, q and dq/dT the matrix for 2M <= n^2
    "n10_m55": (1, lambda: synth.h2_air_mechanism(M=55)),  # one of the two
    "n10_m70": (1, lambda: synth.h2_air_mechanism(M=70)),  # neither
    "n31": (2, lambda: synth.hydrocarbon_mechanism(n_species=30, M=90, n_tb=6, n_troe=4)),
    "n33": (2, lambda: synth.hydrocarbon_mechanism(n_species=32, M=200, n_tb=6, n_troe=4)),
    "n65": (2, lambda: synth.hydrocarbon_mechanism(n_species=64, M=300)),
}


@pytest.mark.parametrize("name", list(MECHS))
def test_layout_edges_match_oracle(name):
    cfg, make = MECHS[name]
    mech = make()
    m, o = df.Mechanism(mech), Mech(mech)
    f = synth.field(cfg, mech, 16, seed=41)
    T, p, Y = _dev(f)
    st, _ = df.integrate(m, T, p, Y, f["dt"], _warp())
    To, Yo, so, _ = o.integrate(f["T"], f["p"], f["Y"], f["dt"])
    assert int(st.abs().sum()) == 0 and np.all(so == 0)
    print(check_integrator(f["T"], f["Y"], T.cpu().numpy(), Y.cpu().numpy(), To, Yo))


@pytest.mark.parametrize("n", [1, 153, 700])
def test_few_cells_bitwise(n):
    """1 to 5 warps per block for these counts, eight for 2000 cells: the same bits."""
    mech = synth.hydrocarbon_mechanism(n_species=16, M=60, n_tb=4, n_troe=2)
    m = df.Mechanism(mech)
    f = synth.field(2, mech, 2000, seed=42)
    T, p, Y = _dev(f)
    Tn, pn, Yn = T[:n].clone(), p[:n].clone(), Y[:, :n].clone()
    df.integrate(m, T, p, Y, f["dt"], _warp())
    df.integrate(m, Tn, pn, Yn, f["dt"], _warp())
    assert torch.equal(T[:n], Tn) and torch.equal(Y[:, :n], Yn)
