"""order_by_T around the cell count below which every cell starts at once and the order
is left out: the same bits with and without it, on both paths."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2210_07094_gb300 as df  # noqa: E402
from paper_2210_07094_gb300 import synth  # noqa: E402

DEV = "cuda:0"


@pytest.mark.parametrize("path,per_sm,extra", [(1, 128, 0), (1, 128, 1), (2, 4, 0), (2, 4, 1)])
def test_order_left_out_below_one_wave(path, per_sm, extra):
    n = per_sm * torch.cuda.get_device_properties(0).multi_processor_count + extra
    mech = synth.h2_air_mechanism()
    m = df.Mechanism(mech)
    f = synth.field(1, mech, n, seed=77)
    res = []
    for order in (1, 0):
        o = df.default_opts()
        o.path, o.order_by_T = path, order
        T, p, Y = (torch.tensor(np.ascontiguousarray(f[k]), device=DEV) for k in ("T", "p", "Y"))
        st, ns = df.integrate(m, T, p, Y, f["dt"], o)
        assert int(st.abs().sum()) == 0
        res.append((T, Y, ns))
    for a, b in zip(*res):
        assert torch.equal(a, b)
