"""The fixed-point near field (P2P variant 1) target by target, where the sizes of the moments differ widely.

theta = 1e-4 leaves every pair in the near field.  One source, two coincident ones of
opposite sign, or one whose potential vanishes at some targets outweigh the others by
2^20 to 2^100: the sums at the heavy particles hold the light ones alone, far below the
scale that the heavy moment sets for the row.
"""
import numpy as np
import pytest

from paper_2005_12351_gb300 import synth
from test_gpu_p2p_fx import LD, evaluate

pytestmark = pytest.mark.gpu

# A pair's term takes about ten roundings of 2^-53 in FP64 arithmetic and fewer in fixed
# point; the sum of up to 300 of them in FP64, of which a thread adds at most a few
# tens in a row, adds as many again: 2^-53 (10 + 20) < 2^-48 of the sum of the magnitudes.
TOL = 2.0 ** -48


def terms(d, D, s):
    """phi and E of sources with moments D (order s) at separations d, one row a source."""
    r2 = (d * d).sum(1)
    y = 1 / np.sqrt(r2)
    y3, y5 = y ** 3, y ** 5
    if s == 0:
        return D[:, 0] * y, (D[:, 0] * y3)[:, None] * d
    if s == 1:
        sr = (D * d).sum(1)
        return -sr * y3, D * y3[:, None] - (3 * sr * y5)[:, None] * d
    G = np.stack([2 * D[:, 0] * d[:, 0] + D[:, 1] * d[:, 1] + D[:, 2] * d[:, 2],
                  D[:, 1] * d[:, 0] + 2 * D[:, 3] * d[:, 1] + D[:, 4] * d[:, 2],
                  D[:, 2] * d[:, 0] + D[:, 4] * d[:, 1] + 2 * D[:, 5] * d[:, 2]], 1)
    q, tr = (G * d).sum(1) / 2, D[:, 0] + D[:, 3] + D[:, 5]
    return 3 * q * y5 - tr * y3, -3 * G * y5[:, None] + (15 * q * y ** 7 - 3 * tr * y5)[:, None] * d


def reference(pos, S, lo, hi):
    """Values at every target and the sums of the magnitudes of the pairs' terms, bounded by those of the
    moments: c |S| / r^(s+1) for the potential (c = 1, 1, 6), c |S| / r^(s+2) for the field (1, 4, 24)."""
    n, P, M = len(pos), pos.astype(LD), S.astype(LD)
    phi, E, mp, me = np.zeros(n, LD), np.zeros((n, 3), LD), np.zeros(n), np.zeros(n)
    for i in range(n):
        d = P[i] - P
        k = (d * d).sum(1) > 0
        o = 0
        for s in range(lo, hi + 1):
            w = (s + 1) * (s + 2) // 2
            D = M[k, o:o + w]
            o += w
            a, b = terms(d[k], D, s)
            phi[i] += a.sum()
            E[i] += b.sum(0)
            r, size = np.sqrt((d[k] ** 2).sum(1)), np.sqrt((D * D).sum(1))
            mp[i] += (1, 1, 6)[s] * float((size / r ** (s + 1)).sum())
            me[i] += (1, 4, 24)[s] * float((size / r ** (s + 2)).sum())
    return phi, E, mp, me


def check(pos, S, lo, hi, leaf, mags=None):
    phi, E, mp, me = reference(pos, S, lo, hi)
    mp, me = (mp, me) if mags is None else mags
    for want in ((True, True), (True, False), (False, True)):
        got = evaluate(pos, S, lo, hi, leaf, 1, want)
        if want[0]:
            assert float((np.abs(got[0] - phi) / mp).max()) < TOL
        if want[1]:
            assert float((np.abs(got[1] - E).max(1) / me).max()) < TOL


SHELLS = [(0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2)]


@pytest.mark.parametrize("lo,hi", SHELLS)
@pytest.mark.parametrize("n,leaf,kind", [(60, 64, "uniform"), (300, 16, "uniform"), (200, 12, "plummer"), (700, 1000, "uniform")])
@pytest.mark.parametrize("ratio", [30, 44, 60, 90])
def test_a_heavy_particle_and_its_neighbours(lo, hi, n, leaf, kind, ratio):
    if n > 300 and ratio != 60:
        pytest.skip("the long row at one ratio")
    pos, S = synth.make_system_mixed(n, lo, hi, kind, 60 + n)
    S[n // 3] *= 2.0 ** ratio
    check(pos, S, lo, hi, leaf)


@pytest.mark.parametrize("lo,hi", SHELLS)
@pytest.mark.parametrize("ratio", [30, 60, 90])
def test_coincident_heavy_particles(lo, hi, ratio):
    """They exclude each other, and at the others their fields cancel (two equal terms of opposite sign)."""
    pos, S = synth.make_system_mixed(120, lo, hi, "uniform", 9)
    pos[40] = pos[80]
    S[40] = 2.0 ** ratio * S[80]
    S[80] = -S[40]
    check(pos, S, lo, hi, 64)


@pytest.mark.parametrize("ratio", [40, 70])
def test_a_heavy_dipole_without_potential_in_its_plane(ratio):
    """A dipole along z gives no potential at the targets of its own z: theirs is the light particles'."""
    pos, S = synth.make_system_mixed(200, 1, 1, "uniform", 13)
    pos[:, 2] = np.where(np.arange(200) % 2 == 0, 0.5, pos[:, 2])
    S[10] = [0.0, 0.0, 2.0 ** ratio]
    phi, E, mp, me = reference(pos, S, 1, 1)
    light = S.copy()
    light[10] = 0.0
    flat = (pos[:, 2] == 0.5) & (np.arange(200) != 10)
    mp[flat] = reference(pos, light, 1, 1)[2][flat]
    check(pos, S, 1, 1, 256, (mp, me))


@pytest.mark.parametrize("lo,hi", SHELLS)
def test_every_size_at_once(lo, hi):
    """Moments spread evenly over 2^-60 to 2^60: many targets of a row fall below its scale."""
    pos, S = synth.make_system_mixed(400, lo, hi, "uniform", 17)
    S = S * 2.0 ** (np.arange(400)[:, None] * 37 % 121 - 60.0)
    check(pos, S, lo, hi, 32)
