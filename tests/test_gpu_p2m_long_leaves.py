"""The FP64 form's P2M over leaves of thousands of particles: its sums restart after 512 of them and lose no bits
with the leaf's length.  The multipoles are those of a Barnes-Hut walk that accepts the root for every target."""
import numpy as np
import pytest

from paper_2005_12351_gb300 import synth
from test_gpu_leaf_expansions import LD, build, indices, mono

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [31, 511, 512, 513, 5000, 100_003])
@pytest.mark.parametrize("lo,hi,p", [(0, 0, 3), (2, 2, 4), (0, 2, 3)])
def test_multipoles_of_one_leaf(n, lo, hi, p):
    import torch
    pos, S = synth.make_system_mixed(n, lo, hi, "uniform", 21 + n)
    S = S * np.where(np.arange(n) % 2 == 0, 1.0, -1.0)[:, None]
    g = build(pos, S, lo, hi, 1 << 20)
    g.evaluate_bh(p, 1e6)
    torch.cuda.synchronize()
    ms = [m for m in indices(p) if sum(m) >= lo]
    al = [a for a in indices(hi) if sum(a) >= lo]
    M = g.copy_array("multipole", len(ms)).numpy()[0]
    centre, half = g.copy_array("centre").numpy().reshape(-1)[:3], float(g.copy_array("half").numpy()[0])
    d, Q = centre.astype(LD) - pos.astype(LD), S.astype(LD)
    big = np.abs(S).max(0)
    for k, m in enumerate(ms):
        ref, size = LD(0), 0.0
        for i, a in enumerate(al):
            q = np.subtract(m, a)
            if q.min() >= 0:
                ref += (mono(d, q) * Q[:, i]).sum()
                size += big[i] * half ** int(q.sum()) / float(np.prod([np.prod(range(1, v + 1)) for v in q]))
        # every product within 2^-56 of its range and the moment's rounding (2^-54), every chunk of 32 within
        # 2^-54, every run of 512 one FP64 rounding of a sum of at most 512
        tol = n * (2.0 ** -56 + 2.0 ** -54) + (n / 32 + 1) * 2.0 ** -54 + (n / 512 + 1) * 512 * 2.0 ** -53
        assert abs(float(M[k] - ref)) <= tol * size, (m, abs(float(M[k] - ref)) / size, tol)
        # the roundings are of both signs: a hundred thousand of them add as a random walk
        if n > 100_000:
            assert abs(float(M[k] - ref)) <= 2.0 ** -41 * size
    g.destroy()
