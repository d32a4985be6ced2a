"""What the speed of this framework is measured on.

Every case is a call (or the few calls) of the public Python binding that a program of this
framework makes, on inputs as it has them in hand: a whole step (load the sources, build the
tree and the lists, evaluate), a repeated evaluation on one geometry, a batch of independent
systems, a burst of requests to the server, a Barnes-Hut step, a Morton order.  The sizes are
those of the repository's configurations, tests and benchmark, or generic ones.

    listed()             the cases
    draw(rng)            one more case of the same ranges
    prepare(case, seed)  inputs and handle, as a program has them before the call
    run(state)           one pass
    work(case)           bytes and flops the path cannot do without
    exact(case, seed)    the FP64 direct sum of the same inputs, in plain torch
"""
import math

import numpy as np
import torch

from paper_2005_12351_gb300 import fmm

# particle pairs of one exact(): a few seconds of FP64 elementwise work
EXACT_PAIRS = 7e10


def _step(name, n, s, p, dist, precision, out, theta=0.5, max_leaf=128, s_hi=None):
    return {"name": name, "kind": "step", "n": n, "s": s, "s_hi": s if s_hi is None else s_hi, "p": p,
            "theta": theta, "max_leaf": max_leaf, "dist": dist, "precision": precision, "out": out}


def listed():
    return [
        # the smallest configuration: a few leaves, where launches and host syncs count
        _step("charges_2k_p4_fp64", 2000, 0, 4, "uniform", "fp64", "both", max_leaf=64),
        # a molecule- or magnet-sized clustered set in the mixed form, odd size
        _step("quadrupoles_12k_plummer_p5_fp32", 12007, 2, 5, "plummer", "fp32", "both", max_leaf=64),
        # an ordinary clustered system in FP64, odd size, high order, adaptive tree
        _step("dipoles_262k_plummer_p8_fp64", 262147, 1, 8, "plummer", "fp64", "both"),
        # the benchmark's step: a million dipoles, the field, FP64
        _step("dipoles_1m_p6_fp64", 1000000, 1, 6, "uniform", "fp64", "field"),
        # the same step in the mixed form
        _step("dipoles_1m_p6_fp32", 1000000, 1, 6, "uniform", "fp32", "field"),
        # the largest single system: four million clustered dipoles on the tensor-core form
        _step("dipoles_4m_plummer_p8_3xtf32", 4000000, 1, 8, "plummer", "3xtf32", "both"),
        # every particle a charge and a dipole (polarisable particles), FP64
        _step("charge_dipole_200k_p6_fp64", 200000, 0, 6, "uniform", "fp64", "both", s_hi=1),
        # a time loop on one geometry: new moments, then the captured evaluate, one graph launch
        {"name": "dipole_loop_125k_p6_fp64", "kind": "loop", "n": 125000, "s": 1, "p": 6, "theta": 0.5,
         "max_leaf": 128, "dist": "uniform", "precision": "fp64", "out": "field"},
        # many independent systems of uneven size as one forest, quadrupoles, FP64
        {"name": "quadrupole_batch_96_p5_fp64", "kind": "batch", "count": 96, "sizes": 1, "n_lo": 256, "n_hi": 65536,
         "s": 2, "p": 5, "theta": 0.5, "max_leaf": 128, "dist": "uniform", "precision": "fp64", "out": "both"},
        # a burst of served requests: host arrays in, host arrays out, four slots
        {"name": "served_burst_16_3xtf32", "kind": "serve", "count": 16, "sizes": 2, "n_lo": 1000, "n_hi": 2000000,
         "slots": 4, "p_lo": 4, "p_hi": 10, "theta": 0.5, "max_leaf": 128, "precision": "3xtf32"},
        # a Barnes-Hut step (charges, potential and field)
        {"name": "barnes_hut_100k_p4", "kind": "bh", "n": 100000, "s": 0, "p": 4, "theta": 0.5, "max_leaf": 128,
         "dist": "uniform", "precision": "fp64", "out": "both"},
        # the Morton order of a point set on its own (load balancing, neighbour search)
        {"name": "morton_1m", "kind": "morton", "n": 1000003, "dist": "plummer"},
    ]


def _log_int(rng, lo, hi):
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return min(hi, max(lo, n | rng.randint(0, 1)))


def draw(rng):
    """One more case: mostly whole steps, as users make them, over the sizes, orders, forms and
    distributions that are listed."""
    kind = rng.choice(["step"] * 6 + ["loop", "batch", "bh", "morton", "serve"])
    dist = rng.choice(["uniform", "plummer"])
    out = rng.choice(["field", "both", "potential"])
    precision = rng.choice(["fp64", "fp64", "fp32", "3xtf32"])
    s = rng.randint(0, 2)
    theta = rng.choice([0.4, 0.5, 0.5, 0.6])
    max_leaf = rng.choice([64, 128])
    if kind == "step":
        n = _log_int(rng, 1000, 1000000 if precision != "fp64" else 600000)
        p = rng.randint(3, 10 if n < 50000 else (8 if n < 300000 else 6))
        s_hi = rng.randint(s, 2) if precision == "fp64" and rng.random() < 0.3 else s
        c = _step("", n, s, p, dist, precision, out, theta, max_leaf, s_hi)
        del c["name"]
        return c
    if kind == "loop":
        return {"kind": "loop", "n": _log_int(rng, 2000, 300000), "s": s, "p": rng.randint(3, 8), "theta": theta,
                "max_leaf": max_leaf, "dist": dist, "precision": precision, "out": out}
    if kind == "batch":
        return {"kind": "batch", "count": rng.randint(12, 90), "sizes": rng.randint(3, 1 << 20), "n_lo": 256,
                "n_hi": _log_int(rng, 2000, 65536), "s": s, "p": rng.randint(3, 6), "theta": theta,
                "max_leaf": max_leaf, "dist": dist, "precision": precision, "out": out}
    if kind == "bh":
        return {"kind": "bh", "n": _log_int(rng, 2000, 150000), "s": s, "p": rng.randint(3, 5),
                "theta": min(theta, 0.5), "max_leaf": max_leaf, "dist": dist, "precision": "fp64", "out": out}
    if kind == "serve":
        return {"kind": "serve", "count": rng.randint(6, 16), "sizes": rng.randint(3, 1 << 20), "n_lo": 1000,
                "n_hi": _log_int(rng, 20000, 1000000), "slots": rng.choice([2, 4]), "p_lo": 4, "p_hi": 8,
                "theta": theta, "max_leaf": max_leaf, "precision": precision}
    return {"kind": "morton", "n": _log_int(rng, 1000, 4000000), "dist": dist}


# ------------------------------------------------------------------- inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) % (1 << 62))


def _positions(n, dist, g):
    """Uniform in the unit cube, or a Plummer sphere of scale radius 0.1 about its middle,
    truncated at ten scale radii (the repository's two distributions)."""
    if dist == "uniform":
        return torch.rand((n, 3), dtype=torch.float64, device="cuda", generator=g)
    x = 10.0
    m = x ** 3 / (1.0 + x * x) ** 1.5 * (1.0 - torch.rand(n, dtype=torch.float64, device="cuda", generator=g))
    r = 0.1 / torch.sqrt(m ** (-2.0 / 3.0) - 1.0)
    u = torch.randn((n, 3), dtype=torch.float64, device="cuda", generator=g)
    u /= u.norm(dim=1, keepdim=True)
    return (0.5 + r[:, None] * u).contiguous()


def _moments(n, s, s_hi, g):
    """Charges in [-1, 1), unit dipoles in random directions, traceless quadrupoles of Gaussian
    tensors (as S_n = Q_n / n!); the orders s..s_hi side by side."""
    parts = []
    for k in range(s, s_hi + 1):
        if k == 0:
            parts.append(2.0 * torch.rand((n, 1), dtype=torch.float64, device="cuda", generator=g) - 1.0)
        elif k == 1:
            u = torch.randn((n, 3), dtype=torch.float64, device="cuda", generator=g)
            parts.append(u / u.norm(dim=1, keepdim=True))
        else:
            a = torch.randn((n, 3, 3), dtype=torch.float64, device="cuda", generator=g)
            q = 0.5 * (a + a.transpose(1, 2))
            tr = (q[:, 0, 0] + q[:, 1, 1] + q[:, 2, 2]) / 3.0
            parts.append(torch.stack([(q[:, 0, 0] - tr) / 2, q[:, 0, 1], q[:, 0, 2], (q[:, 1, 1] - tr) / 2, q[:, 1, 2],
                                      (q[:, 2, 2] - tr) / 2], dim=1))
    return torch.cat(parts, dim=1).contiguous()


def _sizes(case):
    """The systems' sizes and the generator that drew them: the case's own, whatever the inputs' seed."""
    r = np.random.default_rng(case["sizes"])
    lo, hi = math.log(case["n_lo"]), math.log(case["n_hi"])
    # spread over the range in equal steps of its logarithm, one draw from each, in random order
    k = (np.arange(case["count"]) + r.random(case["count"])) / case["count"]
    return r.permutation(np.rint(np.exp(lo + k * (hi - lo))).astype(np.int64)), r


def _system(case, seed):
    """(positions, moments, offsets of the systems) of a case that has them on the GPU."""
    g = _gen(seed)
    if case["kind"] == "batch":
        sizes, _ = _sizes(case)
        off = [0] + [int(v) for v in np.cumsum(sizes)]
    else:
        off = [0, case["n"]]
    pos = _positions(off[-1], case["dist"], g)
    if case["kind"] == "morton":
        return pos, None, off
    return pos, _moments(off[-1], case["s"], case.get("s_hi", case["s"]), g), off


def prepare(case, seed):
    kind = case["kind"]
    if kind == "serve":
        # host arrays, as the clients of a server hold them
        sizes, r = _sizes(case)
        req = []
        for i, n in enumerate(sizes):
            g = _gen(int(seed) * 1009 + i)
            s = int(r.integers(0, 3))
            pos = _positions(int(n), "plummer" if r.random() < 0.5 else "uniform", g).cpu().numpy()
            req.append((pos, _moments(int(n), s, s, g).cpu().numpy(), s, int(r.integers(case["p_lo"], case["p_hi"] + 1))))
        return {"kind": kind, "case": case, "requests": req,
                "server": fmm.Server(slots=case["slots"], precision=case["precision"], mem_budget_bytes=120 << 30)}
    pos, mom, off = _system(case, seed)
    st = {"kind": kind, "case": case, "pos": pos, "mom": mom, "off": off}
    if kind != "morton":
        st["tree"] = fmm.create_tree(max_leaf=case["max_leaf"], precision=case["precision"])
        st["want"] = (case["out"] != "field", case["out"] != "potential")
    if kind == "loop":
        # the geometry is loaded once; the loop brings new moments
        st["tree"].set_sources(pos, mom, case["s"])
    return st


def run(st):
    kind, case = st["kind"], st["case"]
    if kind == "morton":
        return fmm.morton_order(st["pos"])
    if kind == "serve":
        tickets = [st["server"].submit(pos, mom, s, p, theta=case["theta"], max_leaf=case["max_leaf"])
                   for pos, mom, s, p in st["requests"]]
        return [st["server"].wait(t)[:2] for t in tickets]
    tree, (want_phi, want_field) = st["tree"], st["want"]
    if kind == "loop":
        tree.update_moments(st["mom"])
        return tree.evaluate_graph(case["p"], case["theta"], want_phi, want_field)
    if kind == "batch":
        tree.set_sources_batch(st["pos"], st["mom"], st["off"], case["s"])
    elif case.get("s_hi", case["s"]) > case["s"]:
        tree.set_sources_mixed(st["pos"], st["mom"], case["s"], case["s_hi"])
    else:
        tree.set_sources(st["pos"], st["mom"], case["s"])
    if kind == "bh":
        return tree.evaluate_bh(case["p"], case["theta"], want_phi, want_field)
    return tree.evaluate(case["p"], case["theta"], want_phi, want_field)


# --------------------------------------------------------------------- work
def _terms(s, s_hi):
    return sum((k + 1) * (k + 2) // 2 for k in range(s, s_hi + 1))


def _pair_flops(s, s_hi, phi, field):
    """Of one near pair, the root counted once: the shared geometry and each shell's terms."""
    f = 11
    for k in range(s, s_hi + 1):
        f += ((2 if phi else 0) + (7 if field else 0), 5 + (2 if phi else 0) + (15 if field else 0),
              21 + (4 if phi else 0) + (19 if field else 0))[k]
    return f


def _fmm_flops(n, s, s_hi, p, theta, max_leaf, phi, field):
    """A uniform tree's near pairs and M2L (traceless locals and multipoles): the leaves within
    reach of the acceptance criterion, 2/theta half sides, less those outside the box."""
    lev = 0
    while n / 8.0 ** lev > max_leaf:
        lev += 1
    q, side, reach = n / 8.0 ** lev, 2 ** lev, int(1.0 / theta)
    cells = [v for v in ((x, y, z) for x in range(-reach, reach + 1) for y in range(-reach, reach + 1)
                         for z in range(-reach, reach + 1)) if v[0] ** 2 + v[1] ** 2 + v[2] ** 2 <= 1.0 / theta ** 2]
    near = sum(max(0, side - abs(x)) * max(0, side - abs(y)) * max(0, side - abs(z)) for x, y, z in cells) / side ** 3
    m2l = 189.0 * (1.0 / theta / 2.0) ** 3 * n / q if lev >= 2 else 0.0
    tri = lambda k: 2 * k + 1  # noqa: E731
    mac = sum(tri(a) * sum(tri(b) for b in range(s, p + s - a + 1)) for a in range(0 if phi else 1, p + 1))
    return n * q * near * _pair_flops(s, s_hi, phi, field) + 2.0 * mac * m2l


def work(case):
    """Each input read once and each output written once; the method's arithmetic on a uniform set
    of the case's size (a clustered set has about as much)."""
    kind = case["kind"]
    if kind == "morton":
        return {"bytes": case["n"] * 36.0, "flops": 9.0 * case["n"]}
    if kind == "serve":
        sizes = np.exp(np.linspace(math.log(case["n_lo"]), math.log(case["n_hi"]), case["count"]))
        p = (case["p_lo"] + case["p_hi"]) // 2
        return {"bytes": float(sizes.sum()) * 8 * (3 + 3 + 4),
                "flops": sum(_fmm_flops(float(n), 1, 1, p, case["theta"], case["max_leaf"], True, True) for n in sizes)}
    phi, field = case["out"] != "field", case["out"] != "potential"
    s, s_hi = case["s"], case.get("s_hi", case["s"])
    if kind == "batch":
        sizes = np.exp(np.linspace(math.log(case["n_lo"]), math.log(case["n_hi"]), case["count"])).tolist()
    else:
        sizes = [float(case["n"])]
    row = 8 * (3 + _terms(s, s_hi) + int(phi) + 3 * int(field))
    if kind == "bh":
        # about 200 accepted cells and 4 leaves of half-full particles per target
        mul = _terms(s, case["p"])
        flops = case["n"] * (200.0 * mul * 8 + 2.0 * case["max_leaf"] * _pair_flops(s, s_hi, phi, field))
    else:
        flops = sum(_fmm_flops(n, s, s_hi, case["p"], case["theta"], case["max_leaf"], phi, field) for n in sizes)
    return {"bytes": sum(sizes) * row, "flops": flops}


# -------------------------------------------------------------------- exact
def _direct(pos, mom, s, s_hi, phi, field):
    """sum_j over j != i of the sources' potential and E = -grad phi, plain FP64."""
    n = pos.shape[0]
    P = torch.zeros(n, dtype=torch.float64, device="cuda") if phi else None
    E = torch.zeros((n, 3), dtype=torch.float64, device="cuda") if field else None
    rows = max(1, int(2.5e7) // n)
    for a in range(0, n, rows):
        b = min(n, a + rows)
        R = [pos[a:b, k, None] - pos[None, :, k] for k in range(3)]
        r2 = R[0] * R[0] + R[1] * R[1] + R[2] * R[2]
        y = torch.where(r2 > 0, torch.rsqrt(r2), 0.0)
        y2 = y * y
        y3 = y * y2
        col = 0
        for k in range(s, s_hi + 1):
            S = [mom[None, :, col + t] for t in range((k + 1) * (k + 2) // 2)]
            col += len(S)
            if k == 0:
                if phi:
                    P[a:b] += (S[0] * y).sum(1)
                if field:
                    w = S[0] * y3
                    for d in range(3):
                        E[a:b, d] += (w * R[d]).sum(1)
            elif k == 1:
                sr = (S[0] * R[0] + S[1] * R[1] + S[2] * R[2]) * y3
                if phi:
                    P[a:b] -= sr.sum(1)
                if field:
                    w = 3.0 * sr * y2
                    for d in range(3):
                        E[a:b, d] += (S[d] * y3 - w * R[d]).sum(1)
            else:
                G = (2.0 * S[0] * R[0] + S[1] * R[1] + S[2] * R[2], S[1] * R[0] + 2.0 * S[3] * R[1] + S[4] * R[2],
                     S[2] * R[0] + S[4] * R[1] + 2.0 * S[5] * R[2])
                q = 0.5 * (G[0] * R[0] + G[1] * R[1] + G[2] * R[2])
                tr = S[0] + S[3] + S[5]
                y5 = y3 * y2
                if phi:
                    P[a:b] += (3.0 * q * y5 - tr * y3).sum(1)
                if field:
                    w = 15.0 * q * y5 * y2 - 3.0 * tr * y5
                    for d in range(3):
                        E[a:b, d] += (w * R[d] - 3.0 * G[d] * y5).sum(1)
    return P, E


def exact(case, seed):
    kind = case["kind"]
    if kind in ("morton", "serve"):
        return None
    sizes = [case["n"]] if kind != "batch" else _sizes(case)[0].tolist()
    if sum(float(n) ** 2 for n in sizes) > EXACT_PAIRS:
        return None
    pos, mom, off = _system(case, seed)
    phi, field = case["out"] != "field", case["out"] != "potential"
    got = [_direct(pos[a:b], mom[a:b], case["s"], case.get("s_hi", case["s"]), phi, field)
           for a, b in zip(off[:-1], off[1:])]
    return (torch.cat([g[0] for g in got]) if phi else None, torch.cat([g[1] for g in got]) if field else None)
