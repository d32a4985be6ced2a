"""The FP64 form's M2L where the device has no memory for its plan.

FMM_FAIL_SOFT_ALLOC=k (read when a handle is created) fails every allocation of the plan
from the k-th on, as a full device would.  The evaluate then takes the per-cell M2L with
that kernel's bits, and so do later evaluates, captures and replays, which do not try again
before the lists or orders change.
"""
import numpy as np
import pytest

from paper_2005_12351_gb300 import synth
from test_gpu_graph_calls import fresh, host, same

pytestmark = pytest.mark.gpu

N, LEAF, S, P = 120_000, 32, 1, 6


@pytest.mark.parametrize("harmonic", [1, 0])
def test_every_failure_of_a_plan_allocation(monkeypatch, harmonic):
    from gpu_util import to_dev
    from paper_2005_12351_gb300 import fmm
    pos, m1 = synth.make_system(N, S, "uniform", 710)
    X, m1, m2 = to_dev(pos), to_dev(m1), to_dev(m1[::-1].copy())

    def plain(tiled, mom, p=P):
        t = fmm.create_tree(max_leaf=LEAF)
        t.set_tuning(m2l_tiled=tiled, m2l_harmonic=harmonic)
        t.set_sources(X, mom, S)
        out = host(t.evaluate(p, 0.5))
        c = t.launch_count()
        assert same(host(t.evaluate(p, 0.5)), out)
        c, rows = t.launch_count() - c, t.info()["tc_rows"]
        t.destroy()
        assert (rows > 0) == bool(tiled)
        return out, c

    cell, launches = plain(0, m1)
    cell2, _ = plain(0, m2)
    tiles, _ = plain(1, m1)
    cell_up, _ = plain(0, m1, P + 1)
    failed = 0
    for k in range(1, 60):
        monkeypatch.setenv("FMM_FAIL_SOFT_ALLOC", str(k))
        t = fmm.create_tree(max_leaf=LEAF)
        monkeypatch.delenv("FMM_FAIL_SOFT_ALLOC")
        t.set_tuning(m2l_harmonic=harmonic)
        t.set_sources(X, m1, S)
        out = host(t.evaluate(P, 0.5))
        if t.info()["tc_rows"] > 0:            # past the last one
            assert same(out, tiles)
            t.destroy()
            break
        failed += 1
        assert same(out, cell)
        c = t.launch_count()
        assert same(host(t.evaluate(P, 0.5)), cell)
        assert t.launch_count() - c == launches            # not tried again
        assert same(host(t.evaluate_graph(P, 0.5)), cell)
        t.update_moments(m2)
        assert same(host(t.evaluate_graph(P, 0.5)), cell2)
        if k < 4:
            t.update_moments(m1)
            assert same(host(t.evaluate_graph(P + 1, 0.5)), cell_up)       # tried again, fails again
            assert same(host(t.evaluate_graph(P + 1, 0.5)), cell_up)
        t.destroy()
    else:
        assert False, "the plan's allocations did not end"
    assert failed > 10
    assert same(fresh(X, m1, S, "fp64", LEAF, P, 0.5, (True, True)), tiles) or not harmonic
