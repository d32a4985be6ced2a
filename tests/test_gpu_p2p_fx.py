"""The fixed-point near field (P2P variant 1, the FP64 form's default) against a
long-double direct sum, beside the FP64 kernels' error on the same set.

theta = 1e-4 leaves every pair in the near field, so the whole result is the
P2P's.  The sets reach the kernel's edges: one leaf and many, leaves of
different levels in one row (coordinate units change), leaves above the thread
count (tiles), pairs inside and outside the fixed-point range, coincident
points, moments over sixteen decades, zero moments, a set far from the origin
and one at 1e-9 of it.
"""
import numpy as np
import pytest

from paper_2005_12351_gb300 import synth

pytestmark = pytest.mark.gpu

LD = np.longdouble


def direct_ld(pos, S, lo, hi):
    n, P, M = len(pos), pos.astype(LD), S.astype(LD)
    phi, E = np.zeros(n, LD), np.zeros((n, 3), LD)
    for i in range(n):
        R = P[i] - P
        r2 = (R * R).sum(1)
        y = np.where(r2 > 0, 1 / np.sqrt(np.where(r2 > 0, r2, 1)), 0).astype(LD)
        y3, o = y ** 3, 0
        y5, y7 = y3 * y * y, y3 * y ** 4
        for s in range(lo, hi + 1):
            D = M[:, o:o + (s + 1) * (s + 2) // 2]
            o += D.shape[1]
            if s == 0:
                phi[i] += (D[:, 0] * y).sum()
                E[i] += ((D[:, 0] * y3)[:, None] * R).sum(0)
            elif s == 1:
                sr = (D * R).sum(1)
                phi[i] -= (sr * y3).sum()
                E[i] += (D * y3[:, None] - (3 * sr * y5)[:, None] * R).sum(0)
            else:
                G = np.stack([2 * D[:, 0] * R[:, 0] + D[:, 1] * R[:, 1] + D[:, 2] * R[:, 2],
                              D[:, 1] * R[:, 0] + 2 * D[:, 3] * R[:, 1] + D[:, 4] * R[:, 2],
                              D[:, 2] * R[:, 0] + D[:, 4] * R[:, 1] + 2 * D[:, 5] * R[:, 2]], 1)
                q, tr = (G * R).sum(1) / 2, D[:, 0] + D[:, 3] + D[:, 5]
                phi[i] += (3 * q * y5 - tr * y3).sum()
                E[i] += (-3 * G * y5[:, None] + (15 * q * y7 - 3 * tr * y5)[:, None] * R).sum(0)
    return phi, E


def evaluate(pos, S, lo, hi, leaf, variant, want=(True, True), theta=1e-4):
    import torch
    from gpu_util import to_dev
    from paper_2005_12351_gb300 import fmm
    t = fmm.create_tree(max_leaf=leaf)
    t.set_tuning(p2p_variant=variant)
    if hi > lo:
        t.set_sources_mixed(to_dev(pos), to_dev(S), lo, hi)
    else:
        t.set_sources(to_dev(pos), to_dev(S), lo)
    out = t.evaluate(2, theta, *want)
    torch.cuda.synchronize()
    out = [None if v is None else v.cpu().numpy() for v in out]
    t.destroy()
    return out


def rel(a, b):
    return float(np.sqrt(((a.astype(LD) - b) ** 2).sum() / (b ** 2).sum()))


def a_set(n, lo, hi, kind):
    pos, S = synth.make_system_mixed(n, lo, hi, "plummer" if kind in ("levels", "origin", "close") else "uniform", 31 + n)
    if kind == "origin":
        pos = pos - 0.5
    if kind == "offset":
        pos = pos + 1000.0
    if kind == "tiny":
        pos = pos * 1e-9
    if kind == "range":
        S = S * 10.0 ** np.random.default_rng(n).uniform(-8, 8, (n, 1))
        S[::7] = 0.0
    if kind == "close":                       # separations from 2^-1 to 2^-40 of the spacing, and zero
        k = n // 2
        pos[k:2 * k] = pos[:k] + 0.05 * 2.0 ** -np.linspace(1, 40, k)[:, None]
        pos[0] = pos[1]
    return pos, S


@pytest.mark.parametrize("lo,hi", [(0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2)])
@pytest.mark.parametrize("n,leaf,kind", [
    (2, 64, "uniform"), (33, 64, "uniform"), (300, 1000, "uniform"), (300, 16, "levels"), (260, 8, "origin"),
    (260, 16, "offset"), (260, 24, "tiny"), (300, 32, "range"), (200, 12, "close"),
])
def test_error_at_or_below_the_fp64_kernels(lo, hi, n, leaf, kind):
    pos, S = a_set(n, lo, hi, kind)
    ref = direct_ld(pos, S, lo, hi)
    got = evaluate(pos, S, lo, hi, leaf, 1)
    fp64 = evaluate(pos, S, lo, hi, leaf, 2)
    for g, f, r in zip(got, fp64, ref):
        # a rounding of each output and of the coordinates (2^-52) beside the FP64 kernel's own error
        assert rel(g, r) <= 1.5 * rel(f, r) + 2.0 ** -52
    # each output alone gives the same bits
    assert np.array_equal(evaluate(pos, S, lo, hi, leaf, 1, (True, False))[0], got[0])
    assert np.array_equal(evaluate(pos, S, lo, hi, leaf, 1, (False, True))[1], got[1])


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_moments_reach_the_same_targets(bad):
    """A row that holds one falls back to FP64; rows without it stay finite."""
    pos, S = synth.make_system(4000, 1, "uniform", 5)
    S[17, 1] = bad
    for want in ((True, False), (False, True)):
        a = evaluate(pos, S, 1, 1, 16, 1, want, 0.5)
        b = evaluate(pos, S, 1, 1, 16, 0, want, 0.5)
        for x, y in zip(a, b):
            assert (x is None) == (y is None)
            if x is not None:
                assert np.array_equal(np.isfinite(x), np.isfinite(y))
