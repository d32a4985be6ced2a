"""The full Cartesian M2L (m2l_harmonic 0) at the highest orders, whose staged rows barely fit shared memory."""
import numpy as np
import pytest

from paper_2005_12351_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("s,p", [(0, 12), (1, 11), (2, 10), (0, 11)])
@pytest.mark.parametrize("want", [(True, True), (True, False), (False, True)])
def test_against_the_oracle(s, p, want):
    import oracle
    from gpu_util import close, to_dev
    from paper_2005_12351_gb300 import fmm
    pos, S = synth.make_system(3000, s, "uniform", 5)
    S = S.reshape(len(pos), -1)
    t = fmm.create_tree(max_leaf=32)
    t.set_tuning(m2l_harmonic=0)
    t.set_sources(to_dev(pos), to_dev(S), s)
    got = t.evaluate(p, 0.5, *want)
    o = oracle.Tree(pos, 32)
    o.lists(0.5)
    for g, r, w in zip(got, o.fmm(S, s, p), want):
        if w:
            g = g.cpu().numpy()
            assert np.isfinite(g).all() and close(g, r, 1e-12)
    t.destroy()
