"""The FP64 form's expansions at the particles (P2M, M2M, L2P) against extended precision.

Leaves of 1 to 700 particles (the kernels stage 32 at a time and hold 128 threads), the lowest and
highest orders, every instantiation (source terms up to 3, 6 and 10; potential, field, both),
moments over sixteen decades, a set far from the origin, coincident particles.
"""
import math

import numpy as np
import pytest

from paper_2005_12351_gb300 import synth
from test_gpu_m2l_fx import indices

pytestmark = pytest.mark.gpu
LD = np.longdouble
# a displacement, a power and a coefficient are within 2^-56 of their ranges; the
# factors and shifts add FP64 roundings of 2^-53, some thirty on the way up a tree
# of five levels; relative to the sum of the magnitudes of the terms
TOL = 2.0 ** -46


def mono(d, k):
    f = math.prod(math.factorial(q) for q in k)
    return d[..., 0] ** k[0] * d[..., 1] ** k[1] * d[..., 2] ** k[2] / LD(f)


def make(n, s_lo, s_hi, kind, seed):
    pos, _ = synth.make_system(n, 1, "plummer" if kind == "graded" else "uniform", seed)
    S = np.concatenate([synth.make_system(n, s, "uniform", seed + 7 + s)[1].reshape(n, -1)
                        for s in range(s_lo, s_hi + 1)], axis=1)
    if kind == "decades":
        S *= 10.0 ** (16 * synth.uniform01(seed, 3, n) - 8)[:, None]
    if kind == "far":
        pos = pos + np.array([4096.0, -1024.0, 512.0])
    if kind == "same":
        pos[: n // 2] = pos[0]
    return np.ascontiguousarray(pos), np.ascontiguousarray(S)


def build(pos, S, s_lo, s_hi, leaf):
    from gpu_util import to_dev
    from paper_2005_12351_gb300 import fmm
    g = fmm.create_tree(max_leaf=leaf)
    if s_lo == s_hi:
        g.set_sources(to_dev(pos), to_dev(S), s_lo)
    else:
        g.set_sources_mixed(to_dev(pos), to_dev(S), s_lo, s_hi)
    return g


CASES = [(3000, 0, 0, 1, 700, "plain"), (3000, 1, 1, 6, 1, "plain"), (5000, 1, 1, 6, 40, "decades"),
         (4000, 2, 2, 5, 64, "far"), (3000, 0, 1, 6, 150, "graded"), (3000, 0, 2, 8, 33, "plain"),
         (2000, 0, 0, 12, 200, "plain"), (600, 1, 1, 4, 32, "same"), (2, 1, 1, 3, 1, "plain")]


@pytest.mark.parametrize("n,s_lo,s_hi,p,leaf,kind", CASES)
def test_multipoles(n, s_lo, s_hi, p, leaf, kind):
    import torch
    pos, S = make(n, s_lo, s_hi, kind, 40 + p)
    g = build(pos, S, s_lo, s_hi, leaf)
    g.evaluate(p, 0.5)
    torch.cuda.synchronize()
    ms = [m for m in indices(p + s_lo) if sum(m) >= s_lo]
    al = [a for a in indices(s_hi) if sum(a) >= s_lo]
    M = g.copy_array("multipole", len(ms)).numpy()
    rng, centre = g.copy_array("range").numpy(), g.copy_array("centre").numpy()
    perm = g.copy_array("perm").numpy()
    X, Q = pos[perm].astype(LD), S[perm].astype(LD)
    half = g.copy_array("half").numpy()
    worst = 0.0
    for c in range(0, len(rng), max(1, len(rng) // 40)):
        b, e = rng[c]
        d = centre[c].astype(LD) - X[b:e]
        for k, m in enumerate(ms):
            ref, size = LD(0), LD(0)
            for i, a in enumerate(al):
                q = np.subtract(m, a)
                if q.min() >= 0:
                    t = mono(d, q) * Q[b:e, i]
                    ref += t.sum()
                    # a displacement counts as the cell's half side: its rounding does
                    size += (np.abs(Q[b:e, i]) * half[c] ** int(q.sum())
                             / math.prod(math.factorial(v) for v in q)).sum()
            worst = max(worst, float(abs(M[c, k] - ref) / size) if size else abs(M[c, k]))
    print(n, s_lo, s_hi, p, kind, "%.3g" % worst)
    assert worst < TOL * (1 if kind != "far" else 2.0 ** 14)      # centres and positions rounded at 4096
    g.destroy()


@pytest.mark.parametrize("want", [(True, True), (True, False), (False, True)])
@pytest.mark.parametrize("n,s_lo,s_hi,p,leaf,kind", [c for c in CASES if c[0] > 1000 and c[5] != "far"])
def test_evaluation_of_locals(n, s_lo, s_hi, p, leaf, kind, want):
    """phi and E less the near field (its own kernel, tested apart) are the local expansions' values."""
    import torch
    from gpu_util import to_dev
    from paper_2005_12351_gb300 import fmm
    pos, S = make(n, s_lo, s_hi, kind, 40 + p)
    g = build(pos, S, s_lo, s_hi, leaf)
    phi, E = g.evaluate(p, 0.5, *want)
    torch.cuda.synchronize()
    cols = [x for x in indices(p) if x[2] <= 1]
    L = g.copy_array("local", len(cols)).numpy()
    rng, centre, child = g.copy_array("range").numpy(), g.copy_array("centre").numpy(), g.copy_array("child").numpy()
    perm, pairs = g.copy_array("perm").numpy(), g.copy_array("p2p").numpy()
    leaves = np.nonzero(child[:, 1] == 0)[0]
    worst = 0.0
    for c in leaves[:: max(1, len(leaves) // 12)]:
        b, e = rng[c]
        full = {x: LD(v) for x, v in zip(cols, L[c])}
        for x in indices(p):
            if x[2] >= 2:
                full[x] = None
        for z in range(2, p + 1):
            for x in indices(p):
                if x[2] == z:
                    full[x] = -full[(x[0] + 2, x[1], z - 2)] - full[(x[0], x[1] + 2, z - 2)]
        near = np.concatenate([np.arange(*rng[q]) for q in pairs[pairs[:, 0] == c, 1]])
        take = np.arange(b, e)[:: max(1, (e - b) // 8)]
        src = perm[near]
        ph, fe = near_field(pos, S, perm[take], src, s_lo, s_hi)
        d = pos[perm[take]].astype(LD) - centre[c].astype(LD)
        for comp in range(4):
            if not want[0 if comp == 3 else 1]:
                continue
            ref, size = np.zeros(len(take), LD), np.zeros(len(take))
            for k in indices(p if comp == 3 else p - 1):
                x = k if comp == 3 else tuple(v + (i == comp) for i, v in enumerate(k))
                t = mono(d, k) * full[x]
                ref += t
                size += np.abs(t).astype(float)
            got = (phi if comp == 3 else E[:, comp]).cpu().numpy()[perm[take]]
            pn, sz = ph if comp == 3 else (fe[0][comp], fe[1][comp])
            want_v = pn + (ref if comp == 3 else -ref)
            worst = max(worst, float((np.abs(got - want_v) / (size.max() + sz + 1e-300)).max()))
    print(n, s_lo, s_hi, p, kind, want, "%.3g" % worst)
    assert worst < TOL
    g.destroy()


def near_field(pos, S, targets, src, s_lo, s_hi):
    """(phi, magnitude), (E[3], magnitude[3]) of the sources at the targets in long double."""
    from test_gpu_m2l_fx import derivatives
    al = [a for a in indices(s_hi) if sum(a) >= s_lo]
    ph, pm = np.zeros(len(targets), LD), np.zeros(len(targets))
    fe, fm = np.zeros((3, len(targets)), LD), np.zeros((3, len(targets)))
    for i, t in enumerate(targets):
        d = pos[t].astype(LD) - pos[src].astype(LD)
        ok = (d * d).sum(1) > 0
        D = derivatives(d[ok], s_hi + 1)
        for k, a in enumerate(al):
            q = S[src[ok], k].astype(LD)
            v = D[a] * q
            ph[i] += v.sum()
            pm[i] += float(np.abs(v).sum())
            for x in range(3):
                v = D[tuple(np.add(a, [j == x for j in range(3)]).astype(int))] * q
                fe[x, i] -= v.sum()
                fm[x, i] += float(np.abs(v).sum())
    return (ph, pm), (fe, fm)


def test_non_finite_moment_shows():
    import torch
    pos, S = make(3000, 1, 1, "plain", 5)
    S[100, 2] = np.inf
    g = build(pos, S, 1, 1, 40)
    phi, E = g.evaluate(5, 0.5)
    torch.cuda.synchronize()
    assert not np.isfinite(E.cpu().numpy()).any(1).all() and not np.isfinite(phi.cpu().numpy()).all()
    g.destroy()
