"""Particles exactly at their leaf's centre, as on a grid: the local expansion is its first terms there.

Against the oracle, target by target, relative to the sums of the magnitudes of the pairs'
terms: both sides are FP64 evaluations of the same expansions, whose terms are at most some
tens of times those magnitudes in a sum of about a hundred of them.
"""
import numpy as np
import pytest

import oracle
from paper_2005_12351_gb300 import synth
from test_gpu_p2p_heavy import reference

pytestmark = pytest.mark.gpu

TOL = 2.0 ** -53 * 100 * 30


def grid(n, seed):
    """n distinct points of a grid of 16, among them the corner that sets the box."""
    r = np.random.default_rng(seed)
    k = np.concatenate([[0], 1 + r.permutation(16 ** 3 - 1)[: n - 1]])
    return np.stack([k // 256, k // 16 % 16, k % 16], 1) / 16.0


@pytest.mark.parametrize("s,p", [(0, 9), (1, 8), (2, 6)])
@pytest.mark.parametrize("leaf", [1, 3])
@pytest.mark.parametrize("twice", [False, True])
def test_leaves_at_one_point(s, p, leaf, twice):
    from gpu_util import to_dev
    from paper_2005_12351_gb300 import fmm
    pos = grid(300, 3 * s + leaf)
    if twice:
        pos = np.concatenate([pos, pos[::5]])
    S = synth.make_system(len(pos), s, "uniform", 31)[1].reshape(len(pos), -1)
    g = fmm.create_tree(max_leaf=leaf)
    g.set_sources(to_dev(pos), to_dev(S), s)
    phi, E = (v.cpu().numpy() for v in g.evaluate(p, 0.5))
    f1, e1 = g.evaluate(p, 0.5, True, False)[0].cpu().numpy(), g.evaluate(p, 0.5, False, True)[1].cpu().numpy()
    rng, centre, kids = (g.copy_array(a).numpy() for a in ("range", "centre", "child"))
    perm = g.copy_array("perm").numpy()
    at = [(pos[perm[b:e]] == c).all() for (b, e), c, k in zip(rng, centre, kids[:, 1]) if k == 0]
    assert sum(at) > 5                        # the leaves it is about
    t = oracle.Tree(pos, leaf)
    t.lists(0.5)
    phi_o, E_o = t.fmm(S, s, p)
    _, _, mp, me = reference(pos, S, s, s)
    for f in (phi, f1):
        assert float((np.abs(f - phi_o) / mp).max()) < TOL
    for f in (E, e1):
        assert float((np.abs(f - E_o).max(1) / me).max()) < TOL
    g.destroy()
