"""Barnes-Hut targets per warp (8, 16 or 32 by the number of targets): a
system's result has the same bits whichever it is, and meets the oracle's walk
where the warps' queues of cells and leaves fill up and where they hardly do."""
import numpy as np
import pytest
from gpu_util import close

from paper_2005_12351_gb300 import synth

pytestmark = pytest.mark.gpu

TOL = 1e-12        # relative RMS, GPU FP64 vs CPU FP64 oracle, same tree and walk


@pytest.mark.parametrize("s,p,theta,ncrit", [(0, 1, 0.2, 4), (1, 3, 0.5, 32), (2, 4, 0.9, 64)])
def test_same_bits_at_8_16_and_32_targets_per_warp(orc, s, p, theta, ncrit):
    import torch
    from gpu_util import rel_rms, to_dev
    from paper_2005_12351_gb300 import fmm
    sizes = [1, 31, 2500, 33]
    parts = [synth.make_system(n, s, "plummer" if n > 100 else "uniform", 50 + n) for n in sizes]
    got = []
    for total in (0, 70_000, 240_000):          # particles beside them in the batch
        fill = [synth.make_system(total, s, "uniform", 9)] if total else []
        pos = np.concatenate([q[0] for q in parts + fill])
        mom = np.concatenate([q[1] for q in parts + fill])
        off = np.cumsum([0] + [len(q[0]) for q in parts + fill])
        t = fmm.create_tree(max_leaf=ncrit)
        t.set_sources_batch(to_dev(pos), to_dev(mom), off, s)
        phi, E = t.evaluate_bh(p, theta)
        torch.cuda.synchronize()
        n = sum(sizes)
        got.append((phi.cpu().numpy()[:n], E.cpu().numpy()[:n]))
        t.destroy()
    for phi, E in got[1:]:
        assert np.array_equal(phi, got[0][0]) and np.array_equal(E, got[0][1])
    a = 32
    phi_o, E_o = orc.Tree(parts[2][0], ncrit).bh(parts[2][1], s, p, theta)
    assert close(got[0][0][a:a + 2500], phi_o, TOL), rel_rms(got[0][0][a:a + 2500], phi_o)
    assert close(got[0][1][a:a + 2500], E_o, TOL), rel_rms(got[0][1][a:a + 2500], E_o)
