"""A reaction switched off (ln A = -inf): the same bits whether the file or set_lnA says
so, the mechanism's without it to rounding, and back again."""
import copy

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2210_07094_gb300 as df  # noqa: E402
from paper_2210_07094_gb300 import synth  # noqa: E402

N_CELLS = 300


def _run(mech, f, opts):
    T, p, Y = (torch.tensor(np.ascontiguousarray(f[k]), device="cuda") for k in ("T", "p", "Y"))
    dy, q = df.rhs(mech, T, p, Y)
    J = df.jacobian(mech, T, p, Y)
    st, ns = df.integrate(mech, T, p, Y, f["dt"], opts)
    assert not st.any()
    return dy, q, J, T, Y, ns


@pytest.mark.parametrize("cfg,path", [(1, 0), (1, 2), (2, 0)])
def test_reaction_switched_off(cfg, path):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    full = synth.h2_air_mechanism() if cfg == 1 else synth.hydrocarbon_mechanism(n_species=20, M=70, n_tb=4, n_troe=2)
    kinds = [r["type"] for r in full["reactions"]]
    off = [kinds.index("elementary"), kinds.index("three-body"), kinds.index("falloff-troe"), len(kinds) - 1]
    zeroed, without = copy.deepcopy(full), copy.deepcopy(full)
    for j in off:
        zeroed["reactions"][j]["A"] = 0.0
    without["reactions"] = [r for j, r in enumerate(full["reactions"]) if j not in off]
    o = df.default_opts()
    o.path = path
    f = synth.field(cfg, full, N_CELLS, seed=9)
    m, z = df.Mechanism(full), df.Mechanism(zeroed)
    start = _run(m, f, o)
    lnA = torch.tensor([np.log(r["A"]) for r in full["reactions"]], dtype=torch.float64, device="cuda")
    lnA[off] = -np.inf
    m.set_lnA(lnA)
    by_call, by_file = _run(m, f, o), _run(z, f, o)
    for a, b in zip(by_call[:3], by_file[:3]):
        assert torch.equal(a, b)
    m.set_lnA(None)
    for a, b in zip(_run(m, f, o), start):
        assert torch.equal(a, b)
    # without the reactions: the sums have the same terms in the same order
    dy, q, J, T, Y, _ = _run(df.Mechanism(without), f, o)
    scale = lambda a, dims: a.abs().amax(dim=dims, keepdim=True)  # noqa: E731
    assert ((by_call[0] - dy).abs() <= 1e-10 * scale(dy, (0,)).clamp_min(1e-300) + 1e-10 * dy.abs()).all()
    assert ((by_call[2] - J).abs() <= 1e-9 * scale(J, (2,))).all()
    # the integrator's tolerance is 1e-6: two roundings of the same steps
    assert (by_call[3] - T).abs().max() < 1e-6 and (by_call[4] - Y).abs().max() < 1e-9
