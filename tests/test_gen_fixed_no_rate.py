"""Reactions without a rate (A = 0, or a falloff reaction without a low-pressure limit)
keep a mechanism's generated fixed-point evaluation: compared with the FP64 one by the
host build of test_gen_fixed_host, whose driver asks that the states be covered.  (The
mechanism-independent evaluation runs in FP64 then: no temperature is covered there.)"""
import pytest

import test_gen_fixed_host as host


def _without(indices, low=()):
    m = host._forms()
    for j in indices:
        m["reactions"][j]["A"] = 0.0
    for j in low:
        m["reactions"][j]["low"]["A"] = 0.0
    return m


# of _forms' reactions: 0, 2, 4, .. elementary (2, 7 irreversible), 1, 5, 9 third-body, 3, 7 falloff
CASES = {"elementary": ([0], []), "third_body": ([1], []), "falloff": ([3], []), "low_pressure": ([], [7]),
         "several": ([2, 5, 8, 10], [3])}


@pytest.mark.parametrize("name", list(CASES))
def test_no_rate(name, tmp_path, monkeypatch):
    assert "&& mv.T_low < 500" in host.DRIVER
    monkeypatch.setattr(host, "DRIVER", host.DRIVER.replace("&& mv.T_low < 500", "&& mv.T_low == INFINITY"))
    monkeypatch.setitem(host.MECHS, "no_rate", lambda: _without(*CASES[name]))
    host.test_fixed_point_evaluation_matches_fp64("no_rate", tmp_path)
