"""The cell build (one thread-block cluster) bit for bit against the oracle's
tree where its paths change: levels of one cell, of a warp per cell and of
eight lanes per cell, parts of a level that are empty or ragged, chains of
single children that overflow the first cell capacity, several systems."""
import numpy as np
import pytest

from paper_2005_12351_gb300 import synth

pytestmark = pytest.mark.gpu


def pairs(n):
    """n points in pairs 2^-19 of the box apart: long chains of single children."""
    a = synth.make_system(n // 2, 0, "uniform", 71)[0]
    return np.concatenate([a, np.minimum(a + 2.0 ** -19, 1.0 - 2.0 ** -53)])


@pytest.mark.parametrize("kind,n,ncrit", [
    ("uniform", 1, 1), ("uniform", 9, 1), ("plummer", 300, 1), ("uniform", 2049, 8), ("plummer", 40_000, 3),
    ("uniform", 70_000, 1), ("pairs", 1200, 1),
])
def test_cells_are_the_oracles(orc, kind, n, ncrit):
    import torch
    from gpu_util import to_dev
    from paper_2005_12351_gb300 import fmm
    pos = pairs(n) if kind == "pairs" else synth.make_system(n, 0, kind, 600 + n)[0]
    other = synth.make_system(777, 0, "uniform", 5)[0]
    for parts in ([pos], [other, pos, pos[:0], other[:1]]):
        want = [orc.Tree(p, ncrit) if len(p) else None for p in parts]
        allp = np.ascontiguousarray(np.concatenate(parts))
        mom = torch.zeros((len(allp), 1), dtype=torch.float64, device="cuda")
        g = fmm.create_tree(max_leaf=ncrit)
        if len(parts) == 1:
            g.set_sources(to_dev(allp), mom, 0)
        else:
            g.set_sources_batch(to_dev(allp), mom, np.cumsum([0] + [len(p) for p in parts]), 0)
        sysid = g.copy_array("system").numpy()
        arr = {k: g.copy_array(k).numpy() for k in ("level", "coord", "range", "child", "centre", "half", "parent")}
        base = 0
        for s, (p, t) in enumerate(zip(parts, want)):
            if t is None:
                continue
            m = sysid == s
            assert m.sum() == t.ncells
            assert np.array_equal(arr["level"][m], t.level) and np.array_equal(arr["coord"][m], t.ci)
            assert np.array_equal(arr["range"][m], np.stack([t.begin, t.end], 1) + base)
            assert np.array_equal(arr["child"][m][:, 1], t.nchild)
            assert np.array_equal(arr["half"][m], t.halfw)
            if len(parts) == 1:
                assert np.array_equal(arr["child"][:, 0], t.child_first)
                assert np.array_equal(arr["parent"], t.parent)
                assert np.array_equal(arr["centre"], t.centre)
                assert g.info()["nleaves"] == int((t.nchild == 0).sum())
            base += len(p)
        g.destroy()
