"""The numbering of the distinct M2L offsets where its path changes: up to 4,096
of them (ranked by counting), more (radix-sorted), and more than the hash
table starts with.  The lists and the count are checked against the oracle's
lists, the pairs' derivative rows by the FMM result."""
import numpy as np
import pytest
from gpu_util import close, gpu_fmm

from paper_2005_12351_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,dist,ncrit,theta", [
    (3000, "uniform", 64, 0.5), (9000, "plummer", 4, 0.35), (20_000, "uniform", 8, 0.2), (4000, "plummer", 1, 0.1),
])
def test_offsets_are_numbered_by_value(orc, n, dist, ncrit, theta):
    pos, S = synth.make_system(n, 0, dist, 800 + n)
    t = orc.Tree(pos, ncrit)
    t.lists(theta)
    (phi, E), g = gpu_fmm(pos, S, 0, 2, theta, ncrit)
    assert np.array_equal(g.copy_array("m2l").numpy(), t.m2l) and np.array_equal(g.copy_array("p2p").numpy(), t.p2p)
    if len(t.m2l):
        a, b = t.m2l[:, 0], t.m2l[:, 1]
        la, lb = t.level[a].astype(np.int64), t.level[b].astype(np.int64)
        lf = np.maximum(la, lb)
        d = (2 * t.ci[a] + 1) * (1 << (lf - la))[:, None] - (2 * t.ci[b] + 1) * (1 << (lf - lb))[:, None]
        rows = np.column_stack([np.abs(la - lb), la > lb, d])
        assert g.info()["n_doffsets"] == len(np.unique(rows, axis=0))
    phi_o, E_o = t.fmm(S, 0, 2)
    assert close(phi, phi_o, 1e-12) and close(E, E_o, 1e-12)
    g.destroy()
