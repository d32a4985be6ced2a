"""A handle that had to sort a set by all key bits goes back to the leading bits when a set has no long run of ties."""
import numpy as np
import pytest

from paper_2005_12351_gb300 import synth
from test_gpu_tie_sort import points

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [5000, 20_000, 60_000])
def test_the_next_sets_take_the_short_sort_again(orc, n):
    import torch
    from gpu_util import to_dev
    from paper_2005_12351_gb300 import fmm
    ties, flat = points(n, "run1000"), synth.make_system(n, 0, "uniform", 3)[0]
    mom = torch.zeros((n, 1), dtype=torch.float64, device="cuda")
    t = fmm.create_tree(max_leaf=64)
    seen = []
    for pos in (flat, ties, ties, flat, flat):
        c = t.launch_count()
        t.set_sources(to_dev(pos), mom, 0)
        seen.append(t.launch_count() - c)
        o = orc.Tree(pos, 64)
        assert np.array_equal(t.copy_array("keys").numpy().view(np.uint64), o.keys)
        assert np.array_equal(t.copy_array("perm").numpy(), o.perm)
    short, first, again, back, after = seen
    assert first > again > short               # both sorts, then the long one alone
    assert back == again and after == short    # the long one finds no ties: the next is short
    t.destroy()
