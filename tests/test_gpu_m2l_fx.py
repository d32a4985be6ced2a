"""The fixed-point FP64 M2L (m2l_fx.cu) against the sums of Eq. (8) in extended precision."""
import math

import numpy as np
import pytest

from paper_2005_12351_gb300 import synth

pytestmark = pytest.mark.gpu

# Over one target cell, in the cell's own units (L_n h^(|n|+1+s) / n!): the scale
# factors bound the fixed-point sums' error by 2^-55 of the sum over the list of
# max |M'| times the largest row sum of |T'|, which stays within 2^3 of the sum
# of |D_{n+m} M_m| of the low orders; the FP64 rounding of D (2^-53 times the
# recurrence's growth, below 2^4) and of the multipoles' fold (2^-53 times the
# fold's growth, up to 2^|m| <= 2^6 at the orders below) stand beside it.
TOL = 2.0 ** -46


def indices(k):
    return [(x, a - z, z) for q in range(k + 1) for a in range(q + 1) for z in range(a + 1) for x in [q - a]]


def derivatives(v, order):
    """D_k(v), |k| <= order, for rows v of offsets, by the recurrence in long double."""
    d, r2 = {}, (v * v).sum(1)

    def at(k, i, c):
        q = list(k)
        q[i] -= c
        return d[tuple(q)] if q[i] >= 0 else 0

    for k in indices(order):
        if sum(k) == 0:
            d[k] = 1 / np.sqrt(r2)
            continue
        i = next(j for j in range(3) if k[j])
        acc = -(2 * k[i] - 1) * v[:, i] * at(k, i, 1) - (k[i] - 1) ** 2 * at(k, i, 2)
        for j in range(3):
            if j != i and k[j]:
                acc = acc - 2 * k[j] * v[:, j] * at(k, j, 1) - k[j] * (k[j] - 1) * at(k, j, 2)
        d[k] = acc / r2
    return d


def locals_error(g, s, p, want, harmonic=1, count=12):
    """Largest error of L over `count` cells whose ancestors have no list, relative
    to the cell's largest sum of |D M|."""
    ns = [x for x in indices(p) if x[2] <= 1 or not harmonic]
    M = g.copy_array("multipole", len([m for m in indices(p + s) if sum(m) >= s])).numpy()
    L = g.copy_array("local", len(ns)).numpy()
    lists, centre, half = g.copy_array("m2l").numpy(), g.copy_array("centre").numpy(), g.copy_array("half").numpy()
    parent, n = g.copy_array("parent").numpy(), len(centre)
    have = np.bincount(lists[:, 0], minlength=n) > 0
    anc = np.zeros(n, bool)
    for c in range(n):                        # breadth first: parents come before
        if parent[c] >= 0:
            anc[c] = anc[parent[c]] or have[parent[c]]
    free = np.nonzero(have & ~anc)[0]
    ms = [m for m in indices(p + s) if sum(m) >= s]
    worst = 0.0
    for c in free[:: max(1, len(free) // count)][:count]:
        src = lists[lists[:, 0] == c, 1]
        d = derivatives((centre[c] - centre[src]).astype(np.longdouble), p + s)
        err, scale = 0.0, 0.0
        for r, x in enumerate(ns):
            if x[2] > 1 or (sum(x) == 0 and not want[0]):
                continue
            ref, size = np.longdouble(0), 0.0
            for k, m in enumerate(ms):
                if sum(x) + sum(m) <= p + s:
                    t = d[tuple(np.add(x, m))] * M[src, k]
                    ref += t.sum()
                    size += float(np.abs(t).sum())
            w = half[c] ** sum(x) / math.prod(math.factorial(q) for q in x)
            err = max(err, abs(float(ref - L[c, r])) * w)
            scale = max(scale, size * w)
        worst = max(worst, err / scale)
    return worst


# the smallest and largest orders, both parities of the column and multipole
# counts, every dealing of the columns to the warps, both widths of the limbs
# (more than 126 multipoles from p + s = 11 on), the full Cartesian form
@pytest.mark.parametrize("n,leaf,s,p,dist,want,harmonic", [
    (2_200_000, 8, 0, 1, "uniform", (True, True), 1), (1_000_000, 16, 0, 2, "uniform", (True, False), 1),
    (200_000, 16, 1, 4, "uniform", (False, True), 1), (120_000, 16, 1, 6, "uniform", (False, True), 1),
    (60_000, 16, 2, 5, "plummer", (True, True), 1), (60_000, 16, 1, 8, "plummer", (False, True), 1),
    (60_000, 16, 0, 12, "uniform", (True, True), 1), (60_000, 16, 1, 11, "uniform", (False, True), 1),
    (120_000, 16, 1, 5, "uniform", (True, True), 0)])
def test_locals_match_extended_precision(n, leaf, s, p, dist, want, harmonic):
    import torch
    from gpu_util import to_dev
    from paper_2005_12351_gb300 import fmm
    pos, S = synth.make_system(n, s, dist, 900 + p)
    g = fmm.create_tree(max_leaf=leaf)
    g.set_sources(to_dev(pos), to_dev(S), s)
    err, rows = [], []
    for tiled in (0, 1):
        g.set_tuning(m2l_tiled=tiled, m2l_harmonic=harmonic)
        g.evaluate(p, 0.5, *want)
        torch.cuda.synchronize()
        rows.append(g.info()["tc_rows"])
        err.append(locals_error(g, s, p, want, harmonic))
    print(s, p, dist, "FP64 %.3g fixed point %.3g" % tuple(err))
    assert rows[0] == 0 and rows[1] > 0      # the per-cell form, then the tiles
    assert err[1] < TOL
    g.destroy()


def test_routes_agree_and_non_finite_sources_show():
    """One set through the fixed-point form, the per-cell form and a handle with a
    memory budget (which keeps the per-cell form); moments over 200 decades, zero
    moments and a NaN reach the targets they reach in the per-cell form."""
    import torch
    from gpu_util import close, to_dev
    from paper_2005_12351_gb300 import fmm
    pos, S = synth.make_system(130_000, 1, "uniform", 77)
    S[::3] = 0.0
    P = to_dev(pos)

    def run(mom, tiled, budget=0):
        g = fmm.create_tree(max_leaf=32, mem_budget_bytes=budget)
        g.set_tuning(m2l_tiled=tiled)
        g.set_sources(P, to_dev(mom), 1)
        phi, E = g.evaluate(6, 0.5)
        torch.cuda.synchronize()
        rows = g.info()["tc_rows"]
        g.destroy()
        return phi.cpu().numpy(), E.cpu().numpy(), rows

    phi0, E0, r0 = run(S, 0)
    phi1, E1, r1 = run(S, 1)
    phi2, E2, r2 = run(S, 1, 8 << 30)
    assert r0 == 0 and r1 > 0 and r2 == 0
    assert close(E1, E0, 1e-14) and close(phi1, phi0, 1e-14)     # as the P2P variants: FP64 sums in other orders
    assert np.array_equal(E2, E0) and np.array_equal(phi2, phi0)
    for scale in (1e-200, 1e200):
        phi3, E3, _ = run(S * scale, 1)
        assert close(E3 / scale, E1, 1e-15) and close(phi3 / scale, phi1, 1e-15)
    S[12345, 1] = np.nan
    a, b = run(S, 0), run(S, 1)
    assert np.array_equal(np.isfinite(a[1]), np.isfinite(b[1])) and not np.isfinite(b[1]).all()
