"""The scratch of the hottest-first order is there from a mechanism's first call of a size
on, also where that call needed no order: a captured call of the same size under options
that need one allocates nothing."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2210_07094_gb300 as df  # noqa: E402
from paper_2210_07094_gb300 import synth  # noqa: E402


@pytest.mark.parametrize("listed", [False, True])
def test_capture_after_a_call_without_order(listed):
    """128 cells per SM in 32-thread blocks all start at once, in 96-thread blocks 96 do.
    listed: the handle has met a smaller size with an order before."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    n = 128 * torch.cuda.get_device_properties(0).multi_processor_count
    mech = synth.h2_air_mechanism()
    f = synth.field(1, mech, n, seed=3)
    m = df.Mechanism(mech)
    T, p, Y = (torch.tensor(f[k], device="cuda") for k in ("T", "p", "Y"))
    st, ns = torch.zeros((2, n), dtype=torch.int32, device="cuda")
    o, o96 = df.default_opts(), df.default_opts()
    o.jit = o96.jit = 1
    o96.block_threads = 96
    if listed:
        k = n - 1
        df.integrate(m, T[:k].clone(), p[:k].clone(), Y[:, :k].contiguous(), 1e-9, o96)
    T1, Y1 = T.clone(), Y.clone()
    df.integrate(m, T1, p, Y1, 1e-9, o, status=st, nsub=ns)
    T2, Y2 = T.clone(), Y.clone()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        df.integrate(m, T2, p, Y2, 1e-9, o96, status=st, nsub=ns)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(T1, T2) and torch.equal(Y1, Y2) and not st.any()
