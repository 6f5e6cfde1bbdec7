"""The adjoint's separate forward and reverse kernels (stored stages) against
the one kernel that recomputes each step: same arithmetic, so bitwise, at the
edges of a warp, for a mechanism too long for the reverse kernel's theta, and
for cells that fail (non-finite input, more steps than the checkpoints hold)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2210_07094_gb300 as df  # noqa: E402
from paper_2210_07094_gb300 import synth  # noqa: E402

DEV = "cuda:0"


@pytest.mark.parametrize("ncells,M,max_steps,dt_scale", [(1, 25, 32, 1.0), (31, 25, 32, 1.0), (32, 25, 32, 1e-3),
                                                         (33, 25, 4, 1.0), (97, 70, 32, 1.0), (65, 64, 32, 1.0)])
def test_sweeps_apart_match_one_kernel(ncells, M, max_steps, dt_scale):
    mech = synth.h2_air_mechanism(M=M)
    m = df.Mechanism(mech)
    f = synth.field(1, mech, ncells, seed=900 + ncells)
    if ncells > 40:
        f["T"][ncells // 2] = np.nan
    T, p, Y = (torch.tensor(np.ascontiguousarray(f[k]), device=DEV) for k in ("T", "p", "Y"))
    rng = np.random.default_rng(ncells)
    g = [torch.tensor(a, device=DEV) for a in (rng.standard_normal(ncells), rng.standard_normal(Y.shape),
                                               rng.standard_normal(ncells) * 1e-9)]
    full, compact = (df.adjoint(m, T, p, Y, f["dt"] * dt_scale, *g, max_steps=max_steps, store_stages=s)
                     for s in (True, False))
    assert full["workspace"].numel() > compact["workspace"].numel()
    st = full["status"]
    assert set(st.tolist()) <= {0, 1, 2} if ncells > 32 else int(st.abs().sum()) == 0
    for k in ("status", "nsub", "gT0", "gY0", "g_lnA"):
        assert torch.equal(full[k], compact[k]), k
