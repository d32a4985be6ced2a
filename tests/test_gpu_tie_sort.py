"""The Morton sort by leading key bits and the sort of its ties, bit for bit
against the oracle: runs of equal leading bits from one key to past the limit
(256) where the keys go through every pass instead, at the sizes where the
number of passes changes, through each entry point that sorts particles."""
import numpy as np
import pytest

from paper_2005_12351_gb300 import synth

pytestmark = pytest.mark.gpu


def points(n, kind):
    pos = synth.make_system(n, 0, "uniform", 900 + n)[0]
    if kind.startswith("run"):
        # runs of the given length: points that share a cell 2^-14 of the box (past the 39 leading bits), in
        # shuffled order, some of them equal
        m = int(kind[3:])
        k = n // m * m
        base = np.repeat(np.floor(pos[:k // m] * 2.0 ** 14) / 2.0 ** 14, m, axis=0)
        jit = synth.uniform01(77, 1, 3 * k).reshape(k, 3)
        jit[::5] = 0.5
        order = np.argsort(synth.uniform01(78, 2, k), kind="stable")
        pos[:k] = (base + 2.0 ** -15 * jit)[order]
        pos[0], pos[-1] = 0.0, 1.0 - 2.0 ** -53
    return np.ascontiguousarray(pos)


@pytest.mark.parametrize("n,kind", [
    (1, "uniform"), (2, "uniform"), (4096, "run2"), (1 << 14, "run31"), ((1 << 14) + 1, "run33"), (20_000, "run255"),
    (20_001, "run256"), (20_001, "run257"), (60_000, "run1000"), ((1 << 22) + 3, "run7"),
])
def test_order_is_the_oracles(orc, n, kind):
    import torch
    from gpu_util import to_dev
    from paper_2005_12351_gb300 import fmm
    pos = points(n, kind)
    P = to_dev(pos)
    t = orc.Tree(pos, 64)
    outs = [fmm.morton_order(P)]
    if n <= fmm.NOALLOC_MAX_POINTS:
        outs.append((torch.empty_like(outs[0][0]), torch.empty_like(outs[0][1])))
        fmm.morton_order_noalloc(P, *outs[1])
    for keys, perm in outs:
        assert np.array_equal(keys.cpu().numpy().view(np.uint64), t.keys)
        assert np.array_equal(perm.cpu().numpy().astype(np.int64), t.perm)
    tree = fmm.create_tree(max_leaf=64)
    mom = torch.arange(n, dtype=torch.float64, device="cuda").reshape(n, 1)
    # the same handle twice, then on a set without ties
    for p, o in ((P, t), (P, t), (to_dev(points(n, "uniform")), None)):
        tree.set_sources(p, mom, 0)
        if o is not None:
            assert np.array_equal(tree.copy_array("keys").numpy().view(np.uint64), o.keys)
            assert np.array_equal(tree.copy_array("perm").numpy(), o.perm)
            assert np.array_equal(tree.copy_array("range").numpy(), np.stack([o.begin, o.end], 1))
    tree.destroy()


def test_concurrent_calls_share_no_scratch(orc):
    """Morton orders of several threads and streams at once are each their own."""
    import threading
    import torch
    from gpu_util import to_dev
    from paper_2005_12351_gb300 import fmm
    sets = [synth.make_system(30_000 + 1000 * k, 0, "plummer", 40 + k)[0] for k in range(6)]
    want = [orc.Tree(p, 1 << 30) for p in sets]
    bad = []

    def work(k):
        st = torch.cuda.Stream()
        P = to_dev(sets[k])
        torch.cuda.synchronize()
        for _ in range(20):
            keys, perm = fmm.morton_order(P, stream=st)
            if not (np.array_equal(keys.cpu().numpy().view(np.uint64), want[k].keys)
                    and np.array_equal(perm.cpu().numpy().astype(np.int64), want[k].perm)):
                bad.append(k)

    th = [threading.Thread(target=work, args=(k,)) for k in range(len(sets))]
    for t in th:
        t.start()
    for t in th:
        t.join()
    assert not bad
