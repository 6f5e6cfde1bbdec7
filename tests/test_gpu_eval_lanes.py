"""Source terms and Jacobians of few cells run one cell per warp, of more cells one
cell per thread: a cell's bits do not depend on how many share its call, for every
reaction form, inside and outside the fixed-point range of temperatures, and for
states with zeros, negative entries and NaN."""
import copy

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2210_07094_gb300 as df  # noqa: E402
import test_gen_fixed_host as host  # noqa: E402
from paper_2210_07094_gb300 import synth  # noqa: E402


def _forms9():
    """Every reaction form of test_gen_fixed_host with three more (inert) species."""
    m = host._forms()
    for i in range(3):
        m["species"].append(dict(copy.deepcopy(m["species"][i]), name=f"I{i}"))
    return m


MECHS = {"m25": synth.h2_air_mechanism, "m6": lambda: synth.h2_air_mechanism(M=6, n_tb=1, n_troe=1),
         "m70": lambda: synth.h2_air_mechanism(M=70), "forms": _forms9,
         "m0": lambda: dict(synth.h2_air_mechanism(), reactions=[]),
         "third_body": lambda: synth.isomer_mechanism(kind="three-body", A=3e10, eff={"D": 2.5}),
         "irreversible": synth.autocatalytic_mechanism}


@pytest.mark.parametrize("name", list(MECHS))
def test_bits_do_not_depend_on_the_batch(name):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    mech = df.Mechanism(MECHS[name]())
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    N, n = mech.n_species, 16 * sms + 1
    r = np.random.default_rng(7)
    T = r.uniform(300.0, 3500.0, n)
    T[::7] = r.uniform(20.0, 12000.0, T[::7].size)
    Y = 10.0 ** r.uniform(-9.0, 0.0, (N, n))
    Y[r.uniform(size=Y.shape) < 0.05] = 0.0
    Y[r.uniform(size=Y.shape) < 0.05] *= -1e-6
    Y[0] += 1e-3
    Y /= Y.sum(0)
    T[3], Y[1, 4] = np.nan, np.nan
    T, Y = torch.tensor(T, device="cuda"), torch.tensor(Y, device="cuda")
    p = torch.tensor(101325.0 * 10.0 ** r.uniform(-0.3, 1.5, n), device="cuda")
    f, q = df.rhs(mech, T, p, Y)
    J = df.jacobian(mech, T, p, Y)
    assert torch.isfinite(J).float().mean() > 0.9
    same = lambda a, b: bool(((a == b) | (a.isnan() & b.isnan())).all())  # noqa: E731
    for k in (1, 5, 4 * sms, 4 * sms + 1, 16 * sms):
        Tk, pk, Yk = T[:k].clone(), p[:k].clone(), Y[:, :k].clone()
        fk, qk = df.rhs(mech, Tk, pk, Yk)
        Jk = df.jacobian(mech, Tk, pk, Yk)
        assert same(fk, f[:, :k]) and same(qk, q[:k]) and same(Jk, J[:k]), k
