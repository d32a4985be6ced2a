"""Where the FP64 form takes its M2L over target tiles: long lists with many pairs to an offset.

A strongly graded set has thousands of distinct offsets, and the rows of its plan would
hold a few pairs each; it takes the per-cell kernel, whose bits it then has.
"""
import pytest

from paper_2005_12351_gb300 import synth
from test_gpu_graph_calls import host, same

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,n,s,p,theta,tiled", [
    ("plummer", 13_000, 1, 10, 0.5, False),      # 29 pairs an offset
    ("plummer", 18_000, 2, 8, 0.5, False),       # 44
    ("plummer", 20_000, 1, 7, 0.4, False),       # 25
    ("plummer", 60_000, 1, 6, 0.5, True),        # about 150
    ("plummer", 18_000, 1, 11, 0.5, True),       # 44, of the highest orders
    ("plummer", 8_000, 0, 12, 0.5, False),       # 20, of the highest orders
    ("uniform", 20_000, 1, 11, 0.5, True),       # 110, 38,128 pairs
])
def test_route(kind, n, s, p, theta, tiled):
    from gpu_util import to_dev
    from paper_2005_12351_gb300 import fmm
    pos, S = synth.make_system(n, s, kind, 5)
    X, S = to_dev(pos), to_dev(S)
    out = []
    for per_cell in (False, True):
        t = fmm.create_tree(max_leaf=64)
        if per_cell:
            t.set_tuning(m2l_tiled=0)
        t.set_sources(X, S, s)
        out.append(host(t.evaluate(p, theta)))
        info = t.info()
        assert (info["tc_rows"] > 0) == (tiled and not per_cell)
        t.destroy()
    if not tiled:
        assert same(*out)
