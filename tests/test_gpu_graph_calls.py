"""Graph replays between ordinary evaluates of other parameters, and over the FP64 form's fixed-point M2L.

A captured evaluate reads the handle's tables, lists, plan and buffers by address, and an
evaluate of other orders, outputs or theta rewrites or regrows them: the next
evaluate_graph has to capture again.  Every result is a fresh handle's, bit for bit.
"""
import numpy as np
import pytest

from paper_2005_12351_gb300 import synth

pytestmark = pytest.mark.gpu


def host(out):
    import torch
    torch.cuda.synchronize()
    return [None if v is None else v.cpu().numpy().copy() for v in out]


def same(a, b):
    return all((x is None) == (y is None) and (x is None or np.array_equal(x, y)) for x, y in zip(a, b))


def fresh(P, S, s, prec, leaf, p, theta, want):
    from paper_2005_12351_gb300 import fmm
    t = fmm.create_tree(max_leaf=leaf, precision=prec)
    t.set_sources(P, S, s)
    out = host(t.evaluate(p, theta, *want))
    t.destroy()
    return out


# (n, leaf): the FP64 form's per-cell M2L and, at 120,000 points, its tiled one
@pytest.mark.parametrize("prec,n,leaf", [("fp64", 5000, 64), ("fp64", 120_000, 16), ("fp32", 20_000, 32),
                                         ("3xtf32", 20_000, 32)])
def test_replays_between_other_evaluates(prec, n, leaf):
    from gpu_util import to_dev
    from paper_2005_12351_gb300 import fmm
    s, p = 1, 5
    pos, S = synth.make_system(n, s, "uniform", 700)
    P, S = to_dev(pos), to_dev(S)
    t = fmm.create_tree(max_leaf=leaf, precision=prec)
    t.set_sources(P, S, s)
    want = (False, True)
    ref = fresh(P, S, s, prec, leaf, p, 0.5, want)
    assert same(host(t.evaluate_graph(p, 0.5, *want)), ref)
    for q, theta, w in ((p, 0.5, (True, True)), (p + 2, 0.5, want), (p, 0.65, want), (p, 0.5, (True, False)),
                        (p - 2, 0.45, (True, True))):
        assert same(host(t.evaluate(q, theta, *w)), fresh(P, S, s, prec, leaf, q, theta, w))
        for _ in range(2):                    # a capture, then its replay
            assert same(host(t.evaluate_graph(p, 0.5, *want)), ref)
    # an evaluate of the graph's own parameters leaves it in place: one launch
    assert same(host(t.evaluate(p, 0.5, *want)), ref)
    c = t.launch_count()
    assert same(host(t.evaluate_graph(p, 0.5, *want)), ref)
    assert t.launch_count() == c + 1
    t.destroy()


@pytest.mark.parametrize("want", [(True, True), (False, True)])
def test_fixed_point_m2l_in_a_graph(want):
    """Capture, new moments and replay with the FP64 form's M2L over the plan."""
    from gpu_util import to_dev
    from paper_2005_12351_gb300 import fmm
    s, p, leaf = 1, 6, 32
    pos, S1 = synth.make_system(120_000, s, "uniform", 710)
    S2 = S1[::-1].copy()
    P, S1, S2 = to_dev(pos), to_dev(S1), to_dev(S2)
    t = fmm.create_tree(max_leaf=leaf)
    t.set_sources(P, S1, s)
    assert same(host(t.evaluate_graph(p, 0.5, *want)), fresh(P, S1, s, "fp64", leaf, p, 0.5, want))
    assert t.info()["tc_rows"] > 0
    ref = fresh(P, S2, s, "fp64", leaf, p, 0.5, want)
    t.update_moments(S2)
    for _ in range(3):
        assert same(host(t.evaluate_graph(p, 0.5, *want)), ref)
    t.destroy()
