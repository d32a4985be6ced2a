"""A non-finite moment through the FP64 form's expansions alone: the multipoles of its leaf and of every ancestor show
it, those of other cells do not, and every target that its leaf reaches through M2L, and not through the near field, shows
it in the potential and in the field."""
import numpy as np
import pytest

from paper_2005_12351_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("n,leaf,tiled", [(3000, 40, 1), (120_000, 32, 0), (120_000, 32, 1)])
def test_far_targets_and_ancestors(bad, n, leaf, tiled):
    import torch
    from gpu_util import to_dev
    from paper_2005_12351_gb300 import fmm
    pos, S = synth.make_system(n, 1, "uniform", 5 + n)
    S[100, 2] = bad
    g = fmm.create_tree(max_leaf=leaf)
    g.set_tuning(m2l_tiled=tiled)
    g.set_sources(to_dev(pos), to_dev(S), 1)
    phi, E = g.evaluate(6, 0.5)
    torch.cuda.synchronize()
    assert (g.info()["tc_rows"] > 0) == (n > 100_000 and tiled == 1)
    perm, rng, parent = (g.copy_array(k).numpy() for k in ("perm", "range", "parent"))
    child, pairs = g.copy_array("child").numpy(), g.copy_array("p2p").numpy()
    at = int(np.nonzero(perm == 100)[0][0])
    holds = (rng[:, 0] <= at) & (at < rng[:, 1])
    M = g.copy_array("multipole", 119).numpy()               # 1 <= |m| <= 7
    assert np.array_equal(~np.isfinite(M).all(1), holds)
    c = int(np.nonzero(holds & (child[:, 1] == 0))[0][0])
    near = np.zeros(n, bool)
    for a in pairs[pairs[:, 1] == c, 0]:
        near[perm[rng[a, 0]:rng[a, 1]]] = True
    assert 0 < near.sum() < n and parent[c] >= 0
    assert not np.isfinite(phi.cpu().numpy()[~near]).any() and not np.isfinite(E.cpu().numpy()[~near]).any()
    g.destroy()
