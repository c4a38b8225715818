"""The work that programs have this library do, as cases that can be timed.

Every case goes through the public handles (Ecmc, Ecmc.batch, Ecmc3,
EcmcStripes).  A simulation case starts from a melted configuration, loads it
(positions in, overlap check), runs some sweeps and reads positions, counters
and, where the boundary rule has one, the collision pressure back; a
measurement case takes g(r), the hexatic order parameter and the smallest
distance of a configuration.  Case fields:
  kind     cells, batch (many replicas in one handle), cells3 (spheres),
           stripes, measure
  k        disks per side of the start lattice: N = k^2 (k^3 for spheres)
  eta      packing fraction; sigma = 1 throughout
  cells, ell, n_m, sweeps   as for the handles; sweeps = those of one pass
  melt     sweeps from the lattice that prepare() runs
  direction, precision, boundary, lists   the handles' parameters of that name
  host     positions come from and go back to pinned host memory
  tuned    the handle's launch shape is autotuned, as the README does
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1409_6948_gb300 as P
from paper_1409_6948_gb300 import ecmc as E

_MASK = (1 << 64) - 1


def _side(N, eta):
    return math.sqrt(N * math.pi / (4.0 * eta))


def _side3(N, eta):
    return (N * math.pi / (6.0 * eta)) ** (1.0 / 3.0)


def _cells(name, k, eta, cells, ell, n_m, sweeps, melt=20, direction=0, precision=1, boundary=0,
           lists=0, host=False, tuned=False):
    return dict(name=name, kind="cells", k=k, eta=eta, cells=cells, ell=ell, n_m=n_m,
                sweeps=sweeps, melt=melt, direction=direction, precision=precision,
                boundary=boundary, lists=lists, host=host, tuned=tuned)


def listed():
    return [
        # the smallest system of the parity tests: two cells per side, where a
        # sweep is launches and the latency of one chain
        _cells("small", 16, 0.70, 2, 4.0, 2, 10),
        # the paper's Fig. 3 system, N = 256^2: long chains in few, large cells
        _cells("fig3", 256, 0.708, 32, 8.0, 1, 10),
        # the benchmark: a million disks with the paper's choice of parameters,
        # launch shape tuned
        _cells("large", 1024, 0.72, 240, 1.036, 2, 10, tuned=True),
        # the same system driven from the host, one sweep between an upload
        # and a download, as the benchmark's end-to-end figure has it
        _cells("large_host", 1024, 0.72, 240, 1.036, 2, 1, host=True),
        # the largest system of the benchmark
        _cells("huge", 2048, 0.716, 484, 1.053, 2, 2),
        # isotropic chains, which the paper prefers for its applications
        _cells("isotropic", 512, 0.708, 120, 1.06, 2, 4, direction=2),
        # all candidates in FP64: the comparison arm of the FP32 screening
        _cells("fp64", 512, 0.70, 120, 1.20, 2, 4, precision=0),
        # the rejecting boundary rule of Fig. 3, at its many short chains
        _cells("reject", 256, 0.708, 32, 0.25, 16, 10, melt=40, boundary=1),
        # uneven replicas advanced together (the replica scheduler)
        dict(name="replicas", kind="batch", R=96, k_min=64, k_max=512, eta_min=0.60,
             eta_max=0.74, sweeps=4, melt=10),
        # hard spheres at the benchmark's fastest setting
        dict(name="spheres", kind="cells3", k=64, eta=0.45, cells=32, ell=2.0, n_m=1, sweeps=4,
             melt=20),
        # the striped decomposition of Fig. 3
        dict(name="stripes", kind="stripes", k=256, eta=0.708, cells=32, ell=8.0, n_m=1,
             sweeps=4, melt=10, boundary=1, lists=0),
        # the measurements taken between blocks of sweeps
        dict(name="measure", kind="measure", R=1, k=256, eta=0.708, cells=32, rmax=5.0, dr=0.01),
    ]


def _log(rng, a, b):
    return math.exp(rng.uniform(math.log(a), math.log(b)))


def _even(x, least=2):
    return max(least, 2 * int(x / 2.0))


def _nm(per_cell, eta, ell):
    # eq. (nm) of the paper with its mean free path lambda0
    hcp = math.pi / (2.0 * math.sqrt(3.0))
    return max(1, int(math.floor(per_cell * (hcp - eta) / (2.0 * hcp) / ell + 0.5)))


def draw(rng):
    kind = rng.choice(["cells"] * 8 + ["batch"] * 2 + ["cells3"] * 3 + ["stripes"] + ["measure"] * 2)
    if kind == "cells":
        k = int(round(_log(rng, 16, 1024)))
        eta = rng.uniform(0.58, 0.735)
        L = _side(k * k, eta)
        cells = _even(min(L / 2.2, L / _log(rng, 2.2, 9.0)))
        ell = round(_log(rng, 0.25, 8.0), 3)
        nm = _nm(k * k / cells ** 2, eta, ell)
        direction = rng.choice([0, 0, 0, 0, 2])
        boundary = rng.choice([0, 0, 0, 1]) if direction == 0 else 0
        c = _cells("", k, eta, cells, min(ell, 1.0) if boundary else ell, nm,
                   1 + int(rng.random() * (10 if k < 400 else 4)), melt=20, direction=direction,
                   precision=rng.choice([1, 1, 1, 0]), boundary=boundary,
                   host=rng.random() < 0.25)
        del c["name"]
        return c
    if kind == "batch":
        k0 = int(round(_log(rng, 24, 256)))
        k1 = int(round(_log(rng, k0, 512)))
        most = max(1, int(2.5e6 / (0.5 * (k0 * k0 + k1 * k1))))
        return dict(kind=kind, R=min(most, int(round(_log(rng, 2, 128)))), k_min=k0, k_max=k1,
                    eta_min=rng.uniform(0.58, 0.65), eta_max=rng.uniform(0.66, 0.74),
                    sweeps=rng.randint(1, 4), melt=10)
    if kind == "cells3":
        k = int(round(_log(rng, 8, 64)))
        eta = rng.uniform(0.25, 0.48)
        L = _side3(k ** 3, eta)
        cells = _even(L / rng.uniform(2.05, 4.0))
        ell = round(_log(rng, 0.5, 2.0), 3)
        nm = max(1, int(k ** 3 / cells ** 3 * (0.74 - eta) / 2.2 / ell + 0.5))
        return dict(kind=kind, k=k, eta=eta, cells=cells, ell=ell, n_m=nm,
                    sweeps=rng.randint(1, 4), melt=20)
    if kind == "stripes":
        k = int(round(_log(rng, 32, 256)))
        eta = rng.uniform(0.55, 0.72)
        L = _side(k * k, eta)
        return dict(kind=kind, k=k, eta=eta, cells=_even(L / _log(rng, 2.2, 9.0)),
                    ell=round(_log(rng, 1.0, 8.0), 3), n_m=rng.randint(1, 3),
                    sweeps=rng.randint(1, 3), melt=10, boundary=rng.choice([1, 1, 0]),
                    lists=rng.choice([0, 0, 1]))
    k = int(round(_log(rng, 32, 256)))
    eta = rng.uniform(0.58, 0.72)
    L = _side(k * k, eta)
    return dict(kind="measure", R=max(1, min(32, int(rng.random() * 131072 / (k * k)))), k=k,
                eta=eta, cells=_even(L / _log(rng, 3.0, 17.0)), rmax=rng.choice([3.0, 5.0, 6.0]),
                dr=rng.choice([0.01, 0.02]))


# ---- inputs ---------------------------------------------------------------

def _replicas(case, seed):
    """Sizes spread over [k_min, k_max] (over their logarithm), densities in
    turn over the range, cells and chains by the paper's strategy."""
    out = []
    for r in range(case["R"]):
        u = np.random.Generator(np.random.Philox(key=[4, r])).random()
        k = int(round(case["k_min"] * (case["k_max"] / case["k_min"]) ** u))
        eta = case["eta_min"] + (case["eta_max"] - case["eta_min"]) * (r % 29) / 28.0
        L = _side(k * k, eta)
        d = E.suggest_parameters(k * k, L)
        out.append(dict(N=k * k, L=L, cells_x=d["cells_x"], ell=d["ell"], n_m=d["n_m"],
                        seed=seed, replica=r))
    return out


def _disordered(k, eta, seed, rounds=12):
    """k x k disks after Metropolis moves from the square lattice, each disk
    kept within a cage round its site that leaves only the eight neighbouring
    sites in reach; float64 [k, k, 2] in [0, L)."""
    rng = np.random.default_rng(seed)
    L = _side(k * k, eta)
    a = L / k
    cage = min(0.5, a - 0.5 - 1e-6)
    u = np.zeros((k, k, 2))
    i = np.arange(k)
    cls = np.where((k % 2 == 1) & (i == k - 1), 2, i % 2)
    around = [(dy, dx) for dy in (-1, 0, 1) for dx in (-1, 0, 1) if (dy, dx) != (0, 0)]
    kinds = range(3 if k % 2 else 2)
    for _ in range(rounds):
        for p in kinds:
            for q in kinds:
                ys, xs = np.nonzero(cls == p)[0], np.nonzero(cls == q)[0]
                t = u[np.ix_(ys, xs)] + (rng.random((ys.size, xs.size, 2)) - 0.5) * 0.3
                ok = (np.abs(t) <= cage).all(-1)
                for dy, dx in around:
                    v = u[np.ix_((ys + dy) % k, (xs + dx) % k)]
                    d = v - t + np.array([dx * a, dy * a])
                    ok &= (d * d).sum(-1) > 1.0 + 1e-9
                u[np.ix_(ys, xs)] = np.where(ok[..., None], t, u[np.ix_(ys, xs)])
    site = (i + 0.5) * a
    xy = u + np.stack(np.broadcast_arrays(site[None, :], site[:, None]), -1)
    return np.where(xy < 0.0, xy + L, np.where(xy >= L, xy - L, xy))


def _measured(case, seed):
    return np.concatenate([_disordered(case["k"], case["eta"], [seed, r]).ravel()
                           for r in range(case["R"])])


def _handle(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return P.Ecmc.batch(_replicas(case, seed))
    if kind == "cells3":
        h = P.Ecmc3(case["k"] ** 3, _side3(case["k"] ** 3, case["eta"]), 1.0, case["cells"],
                    case["ell"], seed)
        h.set_param(E.PARAM3_N_CHAINS, case["n_m"])
        return h
    N = case["k"] ** 2
    L = _side(N, case["eta"])
    if kind == "stripes":
        h = P.EcmcStripes(N, L, 1.0, case["cells"], case["ell"], seed)
        h.set_param(E.PARAM_STRIPES_N_CHAINS, case["n_m"])
        h.set_param(E.PARAM_STRIPES_BOUNDARY, case["boundary"])
        h.set_param(E.PARAM_STRIPES_LIST_MODE, case["lists"])
        return h
    if kind == "measure":
        return P.Ecmc.batch([dict(N=N, L=L, cells_x=case["cells"], ell=1.0, n_m=1, seed=seed,
                                  replica=r) for r in range(case["R"])])
    h = P.Ecmc(N, L, 1.0, case["cells"], case["cells"], case["ell"], seed)
    h.set_param(E.PARAM_N_CHAINS, case["n_m"])
    for key, name in ((E.PARAM_DIR_MODE, "direction"), (E.PARAM_PRECISION, "precision"),
                      (E.PARAM_BOUNDARY, "boundary"), (E.PARAM_LIST_MODE, "lists")):
        if case[name] != h.get_param(key):
            h.set_param(key, case[name])
    return h


def prepare(case, seed):
    seed = int(seed) & (_MASK >> 1)
    h = _handle(case, seed)
    if case["kind"] == "measure":
        h.set_param(E.PARAM_GR_RMAX, case["rmax"])
        h.set_param(E.PARAM_GR_DR, case["dr"])
        h.set_positions(_measured(case, seed))
        return {"case": case, "h": h}
    h.sweep(case["melt"])
    n = (3 if case["kind"] == "cells3" else 2) * h.N
    if case.get("host"):
        start, out = (torch.empty(n, dtype=torch.float64, pin_memory=True) for _ in range(2))
    else:
        start, out = (torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(2))
    h.positions(start)
    if case.get("tuned"):
        h.autotune()
    return {"case": case, "h": h, "start": start, "out": out}


def _counts(c):
    return np.array([c.sweeps, c.chains, c.events, c.lifts, c.frozen_hits, c.wall_hits,
                     c.rejected_chains], np.int64)


def run(state):
    case, h = state["case"], state["h"]
    if case["kind"] == "measure":
        h.reset_stats()
        h.gr_measure(replica=-1)
        counts = np.stack([h.gr_counts(r)[0] for r in range(case["R"])])
        psi, psi_k, nn, bad = h.hexatic(per_disk=True)
        return (counts, np.atleast_1d(psi), psi_k, nn, bad, np.array([h.min_distance()]))
    h.set_positions(state["start"], case["melt"])
    h.reset_stats()
    h.sweep(case["sweeps"])
    h.positions(state["out"])
    if case["kind"] == "batch":
        p = np.array([h.replica_pressure(r)[0] for r in range(case["R"])])
    elif case.get("boundary"):
        # the pressure of the rejecting rules is read from g(r), not from here
        return (state["out"], _counts(h.counters()))
    else:
        p = np.array([h.pressure()[0]])
    return (state["out"], p, _counts(h.counters()))


# ---- what a pass cannot do without -----------------------------------------

def _rate(eta, dim=2):
    """Contacts of a moving disk (sphere) per sigma: 2 rho g(sigma+) and
    pi rho g(sigma+) with the usual contact values."""
    if dim == 3:
        return 6.0 * eta * (1.0 - 0.5 * eta) / (1.0 - eta) ** 3
    return 8.0 * eta / math.pi * (1.0 - 7.0 * eta / 16.0) / (1.0 - eta) ** 2


def _events(case):
    dim = 3 if case["kind"] == "cells3" else 2
    chains = case["cells"] ** (1 if case["kind"] == "stripes" else dim) * case["n_m"]
    # a chain of the rejecting stripes ends at its first frozen contact, after
    # about a tenth of the contacts that its budget allows
    part = 0.1 if case["kind"] == "stripes" and case["boundary"] else 1.0
    return part * chains * case["ell"] * _rate(case["eta"], dim) * case["sweeps"]


def work(case):
    """Positions in and out once; a contact is decided between about two
    candidates at ten operations each."""
    if case["kind"] == "measure":
        n = case["R"] * case["k"] ** 2
        rho = 4.0 * case["eta"] / math.pi
        bins = int((case["rmax"] - 1.0) / case["dr"] + 0.5)
        pairs = 0.5 * n * rho * math.pi * case["rmax"] ** 2
        return {"bytes": 16.0 * n + 8.0 * case["R"] * bins + 20.0 * n,
                "flops": 10.0 * pairs + 6 * 6 * 10.0 * n}
    if case["kind"] == "batch":
        n, ev = 0, 0.0
        for r, d in enumerate(_replicas(case, 0)):
            eta = case["eta_min"] + (case["eta_max"] - case["eta_min"]) * (r % 29) / 28.0
            n += d["N"]
            ev += d["cells_x"] ** 2 * d["n_m"] * d["ell"] * _rate(eta) * case["sweeps"]
        return {"bytes": 32.0 * n, "flops": 20.0 * ev}
    dim = 3 if case["kind"] == "cells3" else 2
    return {"bytes": 16.0 * dim * case["k"] ** dim, "flops": 20.0 * _events(case)}


# ---- the same results from plain numpy in 64 bits ---------------------------

def _philox(c, k):
    """Philox4x64 with ten rounds (Salmon et al., SC'11)."""
    c0, c1, c2, c3 = c
    k0, k1 = k
    for _ in range(10):
        p0, p1 = 0xD2E7470EE14C6C93 * c0, 0xCA5A826395121157 * c2
        c0, c1, c2, c3 = ((p1 >> 64) ^ c1 ^ k0, p1 & _MASK, (p0 >> 64) ^ c3 ^ k1, p0 & _MASK)
        k0, k1 = (k0 + 0x9E3779B97F4A7C15) & _MASK, (k1 + 0xBB67AE8584CAA73B) & _MASK
    return c0, c1, c2, c3


def _half(v, L):
    return np.where(v >= 0.5 * L, v - L, np.where(v < -0.5 * L, v + L, v))


def _colours(code):
    pool, order = [0, 1, 2, 3], []
    for radix in (6, 2, 1):
        order.append(pool.pop(code // radix))
        code %= radix
    return order + pool


def _chain(a, b, key, member, m, sg, r, extent, reject):
    """One chain in a cell's frame (a along, b across the axis); a is changed
    in place.  Returns (moved, contact sum, counts, accepted)."""
    P0, Q, moved, sum_b = a[m], b[m], [m], 0.0
    ev = lifts = frozen = walls = 0
    before = a.copy() if reject else None
    while True:
        d = sg * (a - P0)
        c2 = (b - Q) * (b - Q)
        hit = (d > 0.0) & (c2 < 1.0)
        hit[m] = False
        j, s = -1, math.inf
        idx = np.nonzero(hit)[0]
        if idx.size:
            ss = np.maximum(0.0, d[idx] - np.sqrt(1.0 - c2[idx]))
            q = np.lexsort((key[idx], ss))[0]
            j, s = idx[q], ss[q]
        sw = max(0.0, extent - P0 if sg > 0 else P0)
        if r <= s and r <= sw:
            a[m] = P0 + sg * r
            return moved, sum_b, (ev, lifts, frozen, walls), True
        if s <= sw:
            ev += 1
            sum_b += d[j] - s
            end, r = P0 + sg * s, r - s
            if member[j]:
                lifts += 1
                a[m] = end
                m = j
                moved.append(m)
                P0, Q = a[m], b[m]
                continue
            frozen += 1
        else:
            walls += 1
            end, r = (extent if sg > 0 else 0.0), r - sw
        if reject:
            a[:] = before
            return [], 0.0, (ev, lifts, frozen, walls), False
        P0, sg = end, -sg


def _sweep(x, y, L, case, seed, t, tot):
    cells, w = case["cells"], L / case["cells"]
    u = _philox((t, 0, 0, 0), (seed, 0))
    sx, sy = ((u[i] >> 11) * 2.0 ** -53 * w for i in (0, 1))
    index = []
    for v, s in ((x, sx), (y, sy)):
        q = v - s
        q = np.where(q < 0.0, q + L, q)
        index.append(np.minimum((q * (1.0 / w)).astype(np.int64), cells - 1))
    cell = index[1] * cells + index[0]
    axis = t & 1
    for colour in _colours((u[2] * 24) >> 64):
        for c in range(cells * cells):
            cx, cy = c % cells, c // cells
            if (cx & 1) + 2 * (cy & 1) != colour:
                continue
            ids = np.nonzero(cell == c)[0]
            if not ids.size:
                continue
            ox, oy = sx + cx * w, sy + cy * w
            X, Y = _half(x - ox, L), _half(y - oy, L)
            others = cell != c
            fx, fy, fk = [X[ids]], [Y[ids]], [ids * 16 + 4]
            for kx in (-1, 0, 1):
                for ky in (-1, 0, 1):
                    XX, YY = X + kx * L, Y + ky * L
                    near = np.nonzero(others & (XX > -1.0) & (XX < w + 1.0) & (YY > -1.0) &
                                      (YY < w + 1.0))[0]
                    fx.append(XX[near])
                    fy.append(YY[near])
                    fk.append(near * 16 + (kx + 1) * 3 + ky + 1)
            fx, fy, key = np.concatenate(fx), np.concatenate(fy), np.concatenate(fk)
            a, b = (fx, fy) if axis == 0 else (fy, fx)
            member = np.arange(a.size) < ids.size
            touched, cell_b = set(), 0.0
            for k in range(case["n_m"]):
                v = _philox((t, 1, c, k), (seed, 0))
                moved, sb, n, kept = _chain(a, b, key, member, (v[0] * ids.size) >> 64,
                                            -1 if v[1] >> 63 else 1, case["ell"], w,
                                            case["boundary"] == 1)
                touched.update(moved)
                cell_b += sb
                tot["n"] += np.array((0, 1) + n + (0 if kept else 1,))
                tot["D"] -= 0.0 if kept else ids.size * case["ell"]
            tot["B"] += ids.size * cell_b
            for j in touched:
                for arr, q, o in ((x, fx, ox), (y, fy, oy)):
                    v = q[j] + o
                    v = v + L if v < 0.0 else v
                    arr[ids[j]] = v - L if v >= L else v
    tot["n"][0] += 1
    tot["D"] += x.size * case["n_m"] * case["ell"]


def _near(xy, L, reach):
    """For chunks of disks: (their indices, separations [m, c, 2] to every
    disk that may lie within reach, which of them are other disks, their
    indices)."""
    N, n = xy.shape[0], max(1, int(L / reach))
    c = np.minimum((xy / L * n).astype(np.int64), n - 1)
    c = c[:, 1] * n + c[:, 0]
    order = np.argsort(c, kind="stable")
    count = np.bincount(c, minlength=n * n)
    first = np.cumsum(count) - count
    table = np.full((n * n, count.max()), -1)
    table[c[order], np.arange(N) - first[c[order]]] = order
    steps = range(-1, 2) if n >= 3 else range(n)
    chunk = max(1, 4000000 // (9 * table.shape[1]))
    for lo in range(0, N, chunk):
        i = np.arange(lo, min(N, lo + chunk))
        cx, cy = c[i] % n, c[i] // n
        j = np.concatenate([table[(cy + dy) % n * n + (cx + dx) % n] for dy in steps
                            for dx in steps], 1)
        yield i, _half(xy[j] - xy[i][:, None], L), (j >= 0) & (j != i[:, None]), j


def _psi(xy, L, rs):
    N = xy.shape[0]
    psi_k, nn, bad = np.zeros(N, complex), np.zeros(N, np.int32), 0
    for i, d, ok, j in _near(xy, L, rs):
        d2 = (d * d).sum(-1)
        ok &= d2 < rs * rs
        m = int(ok.sum(1).max())
        pick = np.argsort(np.where(ok, j, np.iinfo(np.int64).max), axis=1)[:, :m]
        d, d2, ok = (np.take_along_axis(d, pick[..., None], 1), np.take_along_axis(d2, pick, 1),
                     np.take_along_axis(ok, pick, 1))
        lo, hi = np.full(d2.shape, -np.inf), np.full(d2.shape, np.inf)
        for q in range(m):
            # the bisector of disk l, d_l / 2 + t perp(d_l), cut by that of q
            e, e2 = d[:, q:q + 1], d2[:, q:q + 1]
            c = d[..., 0] * e[..., 1] - d[..., 1] * e[..., 0]
            rhs = 0.5 * (e2 - (d * e).sum(-1))
            cut = ok[:, q:q + 1] & (np.arange(m) != q)[None]
            with np.errstate(divide="ignore", invalid="ignore"):
                t = rhs / c
            hi = np.where(cut & (c > 0.0), np.minimum(hi, t), hi)
            lo = np.where(cut & (c < 0.0), np.maximum(lo, t), lo)
            hi = np.where(cut & (c == 0.0) & (rhs < 0.0), -np.inf, hi)
        edge = ok & (hi > lo)
        z = d[..., 0] + 1j * d[..., 1]
        z6 = z * z * z
        z6 = z6 * z6
        z6 = np.where(edge, z6 / np.where(ok, d2, 1.0) ** 3, 0.0)
        nn[i] = edge.sum(1)
        psi_k[i] = z6.sum(1) / np.maximum(nn[i], 1)
        far = np.where(edge, d2 * (0.25 + np.maximum(lo * lo, hi * hi)), 0.0).max(1)
        bad += int((far > 0.25 * rs * rs).sum())
    return psi_k, nn, bad


def exact(case, seed):
    """What run() returns, or None where plain numpy takes too long (event by
    event, some 50 microseconds each).  Isotropic chains have no such value:
    their reflections are chaotic in the last bit."""
    seed = int(seed) & (_MASK >> 1)
    N = case.get("k", 0) ** 2
    L = _side(N, case["eta"]) if N else 0.0
    if case["kind"] == "measure":
        if L < 3.0 * max(case["rmax"], 3.5):
            return None
        all_xy = _measured(case, seed).reshape(case["R"], N, 2)
        bins = int(math.floor((case["rmax"] - 1.0) / case["dr"] + 0.5))
        counts = np.zeros((case["R"], bins), np.int64)
        psi, psi_k, nn, bad, least = [], [], [], 0, 4.0
        for r in range(case["R"]):
            xy = all_xy[r]
            for i, d, ok, _ in _near(xy, L, 1.0 + bins * case["dr"]):
                d2 = d[..., 0] * d[..., 0] + d[..., 1] * d[..., 1]
                d2 = d2[ok]
                least = min(least, d2.min())
                q = (np.sqrt(d2) - 1.0) / case["dr"]
                counts[r] += np.bincount(q[(q >= 0.0) & (q < bins)].astype(np.int64),
                                         minlength=bins)
            pk, n, b = _psi(xy, L, 3.5)
            psi.append(pk.mean())
            psi_k.append(pk)
            nn.append(n)
            bad += b
        return (counts, np.array(psi), np.concatenate(psi_k), np.concatenate(nn), bad,
                np.array([math.sqrt(least)]))
    if case["kind"] != "cells" or case["direction"] != 0 or case["lists"] != 0:
        return None
    total = _events(case) * (case["sweeps"] + case["melt"]) / case["sweeps"]
    if total * (1.0 + N / 4096.0) > 2e5:
        return None
    i = np.arange(N)
    a = L / case["k"]
    x, y = (i % case["k"] + 0.5) * a, (i // case["k"] + 0.5) * a
    tot = {"n": np.zeros(7, np.int64), "B": 0.0, "D": 0.0}
    for t in range(case["melt"] + case["sweeps"]):
        if t == case["melt"]:
            tot = {"n": np.zeros(7, np.int64), "B": 0.0, "D": 0.0}
        _sweep(x, y, L, case, seed, t, tot)
    xy = np.stack([x, y], -1).ravel()
    if case["boundary"]:
        return (xy, tot["n"])
    return (xy, np.array([N / (L * L) * (1.0 + tot["B"] / tot["D"])]), tot["n"])
