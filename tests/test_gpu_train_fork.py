"""The captured training step, whose weight gradients run beside the dZ chain and
whose update writes the bf16 weights itself, against gradient and update as calls of
their own: the same bits, at widths around the update's 32 x 32 tiles; and the bf16
weights are those a reload makes from the master weights."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2210_07094_gb300 as df  # noqa: E402

DEV = "cuda:0"


@pytest.mark.parametrize("widths,n", [((8, 8, 8), 8), ((32, 64, 40), 257), ((200, 24, 136), 1500), ((1600, 800, 400), 512)])
def test_forked_step_matches_separate_calls(widths, n, tmp_path):
    def net():
        o = df.dnn_default_opts()
        o.width[0], o.width[1], o.width[2] = widths
        o.batch = n
        return df.Dnn(o, seed=9)

    g = torch.Generator(device=DEV).manual_seed(n)
    T = 900 + 1500 * torch.rand(n, device=DEV, generator=g, dtype=torch.float64)
    p = 1e5 * (1 + torch.rand(n, device=DEV, generator=g, dtype=torch.float64))
    Y = torch.rand(9, n, device=DEV, generator=g, dtype=torch.float64) + 1e-3
    Y = (Y / Y.sum(0)).contiguous()
    Yn = (Y * (1 + 0.1 * torch.rand(9, n, device=DEV, generator=g, dtype=torch.float64))).contiguous()
    a, b = net(), net()
    for k in (a, b):
        k.fit_norm(T, p, Y, Yn)
    for step in range(4):  # the first as single launches, then the captured graph
        la = a.train_step(T, p, Y, Yn, lr=1e-3)
        lb = b.grad(T, p, Y, Yn)
        b.adam_step(1e-3)
        assert la == lb, step
        assert torch.equal(a.grad_tensor(), b.grad_tensor()), step
        assert np.array_equal(a.params(), b.params()), step
    a.save(str(tmp_path / "net.bin"))
    c = df.Dnn.load(str(tmp_path / "net.bin"))
    assert a.grad(T, p, Y, Yn) == c.grad(T, p, Y, Yn)  # (c has the training scratch from here on, as a has)
    assert torch.equal(a.grad_tensor(), c.grad_tensor())
    X = torch.randn(n, 16, device=DEV, generator=g).to(torch.bfloat16)
    assert torch.equal(a.forward_raw(X), c.forward_raw(X))
