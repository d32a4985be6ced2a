"""The fixed-point near field of leaves at the deepest level that hold more than max_leaf particles: several blocks share
such a leaf's targets.  Counts around a block's two tiles, coincident points and points a billionth apart."""
import numpy as np
import pytest

from paper_2005_12351_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("s,hi", [(0, 0), (1, 1), (0, 2)])
@pytest.mark.parametrize("k", [65, 257, 1025, 3000])
@pytest.mark.parametrize("apart", [0.0, 1e-9])
def test_against_the_direct_sum(s, hi, k, apart):
    import torch
    from gpu_util import to_dev
    from paper_2005_12351_gb300 import fmm
    pos, S = synth.make_system_mixed(1500 + k, s, hi, "uniform", 90 + k)
    pos[1500:] = 0.3 + apart * pos[1500:]
    P, M = to_dev(pos), to_dev(S)
    g = fmm.create_tree(max_leaf=64)
    if hi > s:
        g.set_sources_mixed(P, M, s, hi)
    else:
        g.set_sources(P, M, s)
    phi, E = g.evaluate(2, 1e-4)                 # every pair in the near field
    ref = fmm.direct_sum(P, M, s, source_order_hi=hi)
    torch.cuda.synchronize()
    # two sums of up to 4,500 terms in FP64 or better: 2^-53 of the magnitudes each at every addition
    for a, b in ((phi, ref[0]), (E, ref[1])):
        a, b = a.cpu().numpy().reshape(len(pos), -1), b.cpu().numpy().reshape(len(pos), -1)
        # the magnitude of a target's terms: the pairs inside the heap are the largest, all targets of
        # the heap (and all outside it) have terms of one size
        for part in (slice(0, 1500), slice(1500, None)):
            big = np.abs(b[part]).max()
            assert np.abs(a[part] - b[part]).max() <= 4500 * 2.0 ** -53 * 8 * big
    g.destroy()
