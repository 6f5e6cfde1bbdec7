"""A kernel variant of the generated integrator whose first use falls into the
caller's stream capture: it is compiled, loaded and launched there, as it would be
outside."""
import ctypes as C

import pytest

torch = pytest.importorskip("torch")

import paper_2210_07094_gb300 as df  # noqa: E402
from paper_2210_07094_gb300 import _lib, synth  # noqa: E402

pytestmark = pytest.mark.gpu


def _used(mech):
    used = C.c_int32()
    buf = C.create_string_buffer(512)
    _lib.check(_lib.load().df_chem_jit_info(mech.handle, C.byref(used), buf, 512), "df_chem_jit_info")
    return used.value, buf.value.decode()


@pytest.mark.parametrize("blocking", [False, True])
def test_ignition_variant_first_used_in_a_capture(blocking, monkeypatch):
    """Warmed up with plain substeps only.  blocking: the captured stream is one that the
    legacy stream waits for, so that nothing may be enqueued there meanwhile."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    monkeypatch.setenv("DF_JIT_CACHE", "0")
    mechanism = synth.isomer_mechanism(A=2.0e5, b=0.031 if blocking else 0.032)
    stream = None
    if blocking:
        ptr = C.c_void_p()
        assert C.CDLL("libcudart.so.13").cudaStreamCreate(C.byref(ptr)) == 0
        stream = torch.cuda.ExternalStream(ptr.value)
    n = 40
    T = torch.linspace(900, 1500, n, dtype=torch.float64, device="cuda")
    p = torch.full((n,), 101325.0, dtype=torch.float64, device="cuda")
    Y = torch.zeros((3, n), dtype=torch.float64, device="cuda")
    Y[0], Y[2] = 0.7, 0.3
    tig = torch.zeros(n, dtype=torch.float64, device="cuda")
    st = torch.zeros(n, dtype=torch.int32, device="cuda")
    ns = torch.zeros(n, dtype=torch.int32, device="cuda")
    mech = df.Mechanism(mechanism)
    df.integrate(mech, T.clone(), p, Y.clone(), 1e-6)  # the 32-thread variant, the library's tables
    assert _used(mech)[0] == 1
    Tg, Yg = T.clone(), Y.clone()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        df.integrate_steps(mech, Tg, p, Yg, 1e-6, 3, status=st, nsub=ns, t_ign=tig)
    assert _used(mech)[0] == 1, _used(mech)[1]
    Tg.copy_(T)
    Yg.copy_(Y)
    g.replay()
    torch.cuda.synchronize()
    Te, Ye = T.clone(), Y.clone()
    _, _, te = df.integrate_steps(mech, Te, p, Ye, 1e-6, 3)
    assert _used(mech)[0] == 1
    assert torch.equal(Te, Tg) and torch.equal(Ye, Yg) and torch.equal(te, tig)
    assert not torch.equal(Ye, Y) and not st.any()
