"""Trees with levels of more than 65,536 cells, whose cells the whole chip builds, bit for bit against the oracle:
one such level and several, the last one of leaves only, levels that end at the deepest one, a capacity that
overflows there, more systems than that, and ragged forests."""
import numpy as np
import pytest

from paper_2005_12351_gb300 import synth

pytestmark = pytest.mark.gpu


def points(kind, n):
    pos = synth.make_system(n, 0, "plummer" if kind == "plummer" else "uniform", 800 + n)[0]
    if kind == "pairs":           # long chains of single children, and more cells than the first capacity
        pos = np.concatenate([pos, np.minimum(pos + 2.0 ** -19, 1.0 - 2.0 ** -53)])
    if kind == "same":            # leaves of the deepest level
        pos = np.repeat(pos, 3, axis=0)
    return np.ascontiguousarray(pos)


@pytest.mark.parametrize("kind,n,ncrit", [("uniform", 300_000, 2), ("plummer", 500_000, 1), ("pairs", 80_000, 1),
                                          ("same", 70_000, 2)])
def test_cells_are_the_oracles(orc, kind, n, ncrit):
    import torch
    from gpu_util import to_dev
    from paper_2005_12351_gb300 import fmm
    pos = points(kind, n)
    t = orc.Tree(pos, ncrit)
    assert np.bincount(t.level).max() > 65536
    g = fmm.create_tree(max_leaf=ncrit)
    mom = torch.zeros((len(pos), 1), dtype=torch.float64, device="cuda")
    for _ in range(2):            # the second time with the capacity of the first
        g.set_sources(to_dev(pos), mom, 0)
        arr = {k: g.copy_array(k).numpy() for k in ("level", "coord", "range", "child", "centre", "half", "parent")}
        assert np.array_equal(arr["level"], t.level) and np.array_equal(arr["coord"], t.ci)
        assert np.array_equal(arr["range"], np.stack([t.begin, t.end], 1))
        assert np.array_equal(arr["child"], np.stack([t.child_first, t.nchild], 1))
        assert np.array_equal(arr["parent"], t.parent)
        assert np.array_equal(arr["centre"], t.centre) and np.array_equal(arr["half"], t.halfw)
        assert g.info()["nleaves"] == int((t.nchild == 0).sum()) and g.info()["nlevels"] == int(t.level.max()) + 1
    g.destroy()


def test_more_systems_than_a_wide_level():
    """70,000 systems of 0 to 6 points: the roots are the first wide level.  Each is its own tree."""
    import torch
    from gpu_util import to_dev
    from paper_2005_12351_gb300 import fmm
    sizes = np.arange(70_000) * 5 % 7
    off = np.concatenate([[0], np.cumsum(sizes)])
    pos = synth.make_system(int(off[-1]), 0, "uniform", 8)[0]
    g = fmm.create_tree(max_leaf=2)
    g.set_sources_batch(to_dev(pos), torch.zeros((len(pos), 1), dtype=torch.float64, device="cuda"), off, 0)
    arr = {k: g.copy_array(k).numpy() for k in ("level", "range", "child", "parent", "system")}
    nch, first = arr["child"][:, 1], arr["child"][:, 0]
    assert np.array_equal(arr["range"][:70_000], np.stack([off[:-1], off[1:]], 1))
    count = arr["range"][:, 1] - arr["range"][:, 0]
    split = (count > 2) & (arr["level"] < 21)
    assert np.array_equal(nch > 0, split) and np.all(first[~split] == -1)
    # children follow one another, in order of their parents, and cover their ranges
    kids = np.nonzero(split)[0]
    assert np.array_equal(first[kids], 70_000 + np.concatenate([[0], np.cumsum(nch[kids])[:-1]]))
    for c in kids[:: max(1, len(kids) // 500)]:
        k = np.arange(first[c], first[c] + nch[c])
        assert np.all(arr["parent"][k] == c) and np.all(arr["level"][k] == arr["level"][c] + 1)
        assert np.all(arr["system"][k] == arr["system"][c]) and np.all(count[k] > 0)
        assert arr["range"][k[0], 0] == arr["range"][c, 0] and arr["range"][k[-1], 1] == arr["range"][c, 1]
        assert np.array_equal(arr["range"][k[1:], 0], arr["range"][k[:-1], 1])
    g.destroy()
