"""The fixed-point FP64 M2L against the per-cell kernel at high orders and wide angles, target by target.

The sums over a source's multipoles grow with the order of the local there, so orders need
units of their own.  An FP64 translation is off by a few 2^-53 of the magnitudes of the
pairs' terms; both kernels together by at most 2^-50 of them.
"""
import numpy as np
import pytest

from paper_2005_12351_gb300 import synth
from test_gpu_graph_calls import host

pytestmark = pytest.mark.gpu

TOL = 2.0 ** -50


@pytest.mark.parametrize("s,p,theta,tiled", [(0, 9, 0.6, True), (0, 9, 0.7, True), (1, 8, 0.7, True), (2, 8, 0.7, True),
                                             (0, 10, 0.6, True), (0, 12, 0.5, True), (1, 11, 0.5, True),
                                             (0, 11, 0.6, False), (1, 10, 0.7, False)])
@pytest.mark.parametrize("kind", ["uniform", "plummer"])
@pytest.mark.parametrize("want", [(True, True), (False, True), (True, False)])
def test_each_target(s, p, theta, tiled, kind, want):
    from gpu_util import to_dev
    from paper_2005_12351_gb300 import fmm
    pos, S = synth.make_system(60_000, s, kind, 5)
    S = S.reshape(len(pos), -1)
    t = fmm.create_tree(max_leaf=16)
    t.set_sources(to_dev(pos), to_dev(S), s)
    a = host(t.evaluate(p, theta, *want))
    assert (t.info()["tc_rows"] > 0) == tiled
    t.set_tuning(m2l_tiled=0)
    b = host(t.evaluate(p, theta, *want))
    t.destroy()
    size = np.sqrt((S ** 2).sum(1))
    for x, y, q, c in ((a[0], b[0], 1, (1, 1, 6)[s]), (a[1], b[1], 2, (1, 4, 24)[s])):
        if x is None:
            continue
        d = np.abs(x - y).reshape(len(pos), -1).max(1)
        for j in np.argsort(-d)[:40]:                   # the targets furthest off
            r2 = ((pos - pos[j]) ** 2).sum(1)
            r2[r2 == 0] = np.inf
            assert d[j] <= TOL * c * (size * r2 ** (-(s + q) / 2)).sum()
