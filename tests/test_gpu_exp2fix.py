"""The fixed-point exponential of the rate expressions against the host libm."""
import ctypes as C

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("top", [1e-300, 2.0 ** -53, 1e-6, 1.0, 64.0, 511.999, 800.0])
def test_exp_rate(top):
    """Error bound: the argument's floor 0.35 ulp of a result just above a power
    of two (0.7 just below), the rounding 0.5, the truncated products and the
    polynomial below 0.1, for |x| >= 128 the reduction's two units 0.35 more:
    1.6 ulp, and half an ulp for the host's exp.  Beyond |x| = 512 the library exp
    (1 ulp), subnormal results and overflow included."""
    from paper_2210_07094_gb300 import _lib
    L = _lib.load()
    rng = np.random.default_rng(7)
    x = np.concatenate([rng.uniform(-top, top, 1 << 18), [0.0, -0.0, top, -top, np.nextafter(512.0, 0), 512.0, -512.0,
                                                          5e-324, -5e-324, np.inf, -np.inf, np.nan]])
    xd = torch.tensor(x, device="cuda")
    yd = torch.empty_like(xd)
    _lib.check(L.df_probe_exp_rate(C.c_void_p(xd.data_ptr()), C.c_void_p(yd.data_ptr()), x.size,
                                   C.c_void_p(torch.cuda.current_stream().cuda_stream)), "df_probe_exp_rate")
    y = yd.cpu().numpy()
    with np.errstate(over="ignore", under="ignore"):
        ref = np.exp(x)
    fin = np.isfinite(ref)
    assert np.array_equal(y[~fin & ~np.isnan(ref)], ref[~fin & ~np.isnan(ref)]) and np.isnan(y[-1])
    assert np.max(np.abs(y[fin] - ref[fin]) / np.spacing(ref[fin])) <= 2.1
    assert y[1 << 18] == 1.0 and y[(1 << 18) + 1] == 1.0
