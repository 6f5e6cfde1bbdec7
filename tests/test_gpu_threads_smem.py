"""Calls of different sizes from two threads, each with a handle and a stream of its own:
the launches of one kernel with little and with much shared memory do not take each
other's room (a launch beyond the kernel's limit is refused by the runtime)."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2210_07094_gb300 as df  # noqa: E402
from paper_2210_07094_gb300 import synth  # noqa: E402


def _both(calls, repeats):
    """Every callable repeats times in a thread of its own, started together."""
    errors, gate = [], threading.Barrier(len(calls))

    def work(call):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                gate.wait()
                for _ in range(repeats):
                    call()
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    ts = [threading.Thread(target=work, args=(c,)) for c in calls]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors[0]


def _cells(cfg, mech, n):
    f = synth.field(cfg, mech, n, seed=n)
    return [torch.tensor(np.ascontiguousarray(f[k]), device="cuda") for k in ("T", "p", "Y")]


def test_warp_integrator_of_few_and_many_cells():
    """64 cells of 50 species take a warp (28 KB) per block, 1300 all the shared memory."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    mech = synth.hydrocarbon_mechanism()
    calls = []
    for n in (64, 1300):
        m = df.Mechanism(mech)
        T, p, Y = _cells(2, mech, n)
        st, ns = torch.zeros((2, n), dtype=torch.int32, device="cuda")
        o = df.default_opts()
        o.max_substeps = 1  # one attempt: the launches, not the kernels, set the time
        calls.append(lambda m=m, T=T, p=p, Y=Y, st=st, ns=ns, o=o: df.integrate(m, T, p, Y, 1e-9, o, status=st, nsub=ns))
        calls[-1]()
    _both(calls, 400)


def test_source_terms_and_jacobians_of_few_and_more_cells():
    """One warp per block up to a cell per SM, four from four: 9 species, 300 reactions."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    mech = synth.h2_air_mechanism()
    mech = dict(mech, reactions=mech["reactions"] * 12)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    calls = []
    for n in (sms, 4 * sms):
        m = df.Mechanism(mech)
        T, p, Y = _cells(1, mech, n)
        calls.append(lambda m=m, T=T, p=p, Y=Y: (df.rhs(m, T, p, Y), df.jacobian(m, T, p, Y)))
        calls[-1]()
    _both(calls, 400)
