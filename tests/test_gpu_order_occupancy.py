"""The hottest-first order is left out only where the launch that follows really starts
every cell at once, one warp per FP64 pipe: counted as the nodes of a captured call (the
order is four of them) around the line, for launches of which an SM holds fewer than
four warps, by the sizes of their shared memory."""
import ctypes as C

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2210_07094_gb300 as df  # noqa: E402
from paper_2210_07094_gb300 import synth  # noqa: E402


def _nodes(m, f, n, o):
    """Graph nodes of one df.integrate of n cells (run once before: allocations)."""
    rt = C.CDLL("libcudart.so.13")
    T, p, Y = (torch.tensor(np.ascontiguousarray(f[k][..., :n]), device="cuda") for k in ("T", "p", "Y"))
    st, ns = torch.zeros((2, n), dtype=torch.int32, device="cuda")
    df.integrate(m, T, p, Y, 1e-9, o, status=st, nsub=ns)
    torch.cuda.synchronize()
    stream, graph, count = C.c_void_p(), C.c_void_p(), C.c_size_t()
    assert rt.cudaStreamCreateWithFlags(C.byref(stream), 1) == 0
    assert rt.cudaStreamBeginCapture(stream, 2) == 0
    try:
        df.integrate(m, T, p, Y, 1e-9, o, status=st, nsub=ns, stream=torch.cuda.ExternalStream(stream.value))
    finally:
        rc = rt.cudaStreamEndCapture(stream, C.byref(graph))
    assert rc == 0 and rt.cudaGraphGetNodes(graph, None, C.byref(count)) == 0
    rt.cudaGraphDestroy(graph)
    rt.cudaStreamDestroy(stream)
    return count.value


def _times(mech, k):
    return dict(mech, reactions=mech["reactions"] * k)


# mechanism, options, cells per SM up to which the order is left out: 228 KB of shared
# memory per SM over 52.5 KB per 32 cells and the staged mechanism (9 species), 227 KB over
# a warp's share (50 species)
H2, CHON = synth.h2_air_mechanism, synth.hydrocarbon_mechanism
CASES = {"generated": (1, H2, {}, 128),
         "blob": (1, H2, {"jit": 1}, 128),                                  # 2.7 KB staged: 4 blocks
         "blob_100_reactions": (1, lambda: _times(H2(), 4), {"jit": 1}, 96),     # 7.4 KB: 3
         "volume_500_reactions": (1, lambda: _times(H2(), 20), {"reactor": 1}, 64),  # 32 KB: 2
         "block_96": (1, H2, {"jit": 1, "block_threads": 96}, 96),
         "one_block_per_sm": (1, H2, {"block_threads": 32, "blocks_per_sm": 1}, 32),
         "warp": (2, CHON, {}, 4),
         "warp_1800_reactions": (2, lambda: _times(CHON(), 6), {}, 2)}     # 85 KB a cell


@pytest.mark.parametrize("name", list(CASES))
def test_order_where_cells_wait(name):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    cfg, make, opts, per_sm = CASES[name]
    line = per_sm * torch.cuda.get_device_properties(0).multi_processor_count
    mech = make()
    m = df.Mechanism(mech)
    f = synth.field(cfg, mech, line + 1, seed=5)
    o = df.default_opts()
    for k, v in opts.items():
        setattr(o, k, v)
    assert _nodes(m, f, line + 1, o) == _nodes(m, f, line, o) + 4
    o.order_by_T = 0
    assert _nodes(m, f, line + 1, o) == _nodes(m, f, line, o)
