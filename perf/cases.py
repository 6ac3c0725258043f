"""Performance cases of the P3T long-range force on one GPU.

One pass of a case is what an integrator asks of the library once per
long-range (tree) step: rebuild the tree over the moved particles, walk it,
evaluate accelerations and potentials and return the r_out neighbour lists;
or the same for a batch of clusters, the orbit-dependent neighbour search on
a built tree, or the tidal-tensor measurement of a set of binaries.  Device
tensors in, device tensors out, with the tree handle, the context and the
output buffers kept from step to step as a program keeps them.

The float64 results of PT_MIXED carry float32 pair arithmetic (errors of
~1e-7), so its cases return them as float32, the type that says how much of
them is meant; PT_FP64 results stay float64.

``exact`` evaluates the same tree method (same root box, keys, octree,
groups, acceptance test and changeover) with plain torch float64 operations,
so that it agrees with the library to rounding, not only to the tree's
truncation error.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2006_16560_gb300 import binding as B

DEV = "cuda"
PLUMMER_A = 3.0 * math.pi / 16.0
AU = 4.84813681109536e-06 * 0.7686          # 1 AU for a half-mass radius of 1 pc, Henon units

# The tree parameters of the repository's configurations: the headline
# quadrupole setup (theta 0.3, 16 particles per leaf, 64 per group) and the
# small monopole one (theta 0.5, 8 per leaf).
QUAD = {"order": 2, "theta": 0.3, "n_leaf": 16, "n_group": 64}
MONO = {"order": 0, "theta": 0.5, "n_leaf": 8, "n_group": 64}


def _step(name, n, precision, masses="kroupa", md=0, r_out=0.003, **tree):
    return {"name": name, "kind": "step", "n": n, "precision": precision, "masses": masses, "md": md,
            "r_out": r_out, **tree}


def listed():
    return [
        # a small open cluster, stepped by a laptop-sized run: launches and latency
        _step("step_1000", 1000, "mixed", "equal", r_out=0.05, **MONO),
        # the plain float64 validation configuration (4,096 equal masses, monopole)
        _step("fp64_4096", 4096, "fp64", "equal", r_out=0.05, **MONO),
        # globular clusters in mixed precision, from the smallest size at which a tree pays
        # to the headline million and the ten-million set (sizes not multiples of anything)
        _step("step_16k", 16384, "mixed", **QUAD),
        _step("step_100k", 100003, "mixed", **QUAD),
        _step("step_1m", 1048576, "mixed", **QUAD),
        _step("step_10m", 10000000, "mixed", **QUAD),
        # the float64 path on the headline tree parameters
        _step("fp64_150k", 150001, "fp64", **QUAD),
        # every star in a Kroupa (1995) binary, mass-dependent changeover radii
        _step("binaries_400k", 400000, "mixed", "binaries", 1, 0.00199039 * 2.5 ** (1 / 3), **QUAD),
        # an ensemble of independent clusters in one replayed launch sequence
        {"name": "batch_256", "kind": "batch", "sets": 256, "nmin": 1024, "nmax": 65536, "precision": "mixed",
         "order": 2, "theta": 0.4, "n_leaf": 16, "n_group": 64},
        # a handful of small clusters, as a server's light load puts them together
        {"name": "batch_12", "kind": "batch", "sets": 12, "nmin": 600, "nmax": 6000, "precision": "mixed",
         "order": 2, "theta": 0.4, "n_leaf": 8, "n_group": 64},
        # the short-range integrator's neighbour search with velocities (Eq. 24)
        {"name": "orbit_250k", "kind": "orbit", "n": 250007, "masses": "kroupa", "md": 0,
         "r_out": 0.2 * 250007 ** (-1 / 3), "precision": "mixed", **QUAD},
        # tidal tensors of binaries: measure points through the float64 force, fit, evaluation
        {"name": "tidal_24k", "kind": "tidal", "n": 24000, "bins": 2500, "tidal_order": 2, "masses": "kroupa",
         "md": 0, "r_out": 0.2 * 24000 ** (-1 / 3), "precision": "fp64", **QUAD},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["mixed", "mixed", "mixed", "mixed", "fp64", "fp64", "binaries", "batch", "orbit", "tidal"])
    tree = {"order": rng.choice([0, 2, 2, 2]), "theta": round(rng.uniform(0.3, 0.6), 3),
            "n_leaf": rng.choice([8, 12, 16]), "n_group": rng.choice([32, 48, 64, 64, 64])}
    if kind == "batch":
        nmin = _log_uniform(rng, 500, 4000)
        return {"kind": "batch", "sets": _log_uniform(rng, 4, 256), "nmin": nmin,
                "nmax": nmin * rng.choice([2, 4, 16]), "precision": "mixed", **tree}
    n = _log_uniform(rng, 1000, {"mixed": 3000000, "fp64": 150000, "binaries": 400000, "orbit": 250000,
                                 "tidal": 24000}[kind])
    c = {"kind": "step", "n": n, "precision": "mixed", "masses": rng.choice(["equal", "kroupa"]),
         "md": 0, "r_out": rng.uniform(0.1, 0.4) * n ** (-1 / 3), **tree}
    if kind == "mixed":
        c["md"] = rng.choice([0, 0, 0, 1])
    elif kind == "fp64":
        c["precision"] = "fp64"
        c["md"] = rng.choice([0, 0, 0, 1])
    elif kind == "binaries":
        c.update(n=n + n % 2, masses="binaries", md=rng.choice([0, 1]))
    elif kind == "orbit":
        c.update(kind="orbit", md=rng.choice([0, 1]))
    elif kind == "tidal":
        c.update(kind="tidal", bins=max(1, n // rng.choice([10, 30])), tidal_order=2, precision="fp64", masses="kroupa")
    return c


# ---- inputs ----------------------------------------------------------------

def _iso(g, n):
    z = 2 * torch.rand(n, generator=g, device=DEV, dtype=torch.float64) - 1
    p = 2 * math.pi * torch.rand(n, generator=g, device=DEV, dtype=torch.float64)
    s = torch.sqrt(1 - z * z)
    return torch.stack([s * torch.cos(p), s * torch.sin(p), z], 1)


def _kroupa(g, n, mmax=150.0):
    """Kroupa (2001) masses (slopes 1.3 / 2.3, break 0.5 Msun, from 0.08), solar units."""
    u = torch.rand(n, generator=g, device=DEV, dtype=torch.float64)
    i1 = (0.08 ** -0.3 - 0.5 ** -0.3) / 0.3
    i2 = 0.5 * (0.5 ** -1.3 - mmax ** -1.3) / 1.3
    u = u * (i1 + i2)
    low = (0.08 ** -0.3 - 0.3 * u.clamp(max=i1)).pow(-1 / 0.3)
    high = (0.5 ** -1.3 - 1.3 * (u - i1).clamp(min=0) / 0.5).pow(-1 / 1.3)
    return torch.where(u < i1, low, high)


def _plummer(g, n):
    """Plummer sphere in Henon units (truncated at mass fraction 0.999): positions, velocities."""
    x = torch.rand(n, generator=g, device=DEV, dtype=torch.float64) * 0.999 + 1e-12
    r = PLUMMER_A / torch.sqrt(x.pow(-2 / 3) - 1)
    # speeds: q = v / v_esc, density q^2 (1 - q^2)^3.5, by inverting its tabulated distribution
    q = torch.linspace(0, 1, 4097, device=DEV, dtype=torch.float64)
    cdf = torch.cumsum(q * q * (1 - q * q) ** 3.5, 0)
    u = torch.rand(n, generator=g, device=DEV, dtype=torch.float64) * cdf[-1]
    k = torch.searchsorted(cdf, u).clamp(1, 4096)
    v = q[k - 1] + (u - cdf[k - 1]) / (cdf[k] - cdf[k - 1]) / 4096
    v = v * math.sqrt(2 / PLUMMER_A) * (1 + (r / PLUMMER_A) ** 2) ** -0.25
    return _iso(g, n) * r[:, None], _iso(g, n) * v[:, None]


def _binaries(g, pairs):
    """Every star in a binary: Kroupa (1995) periods, thermal eccentricities (particles 2k, 2k + 1)."""
    cen, vel = _plummer(g, pairs)
    m = _kroupa(g, 2 * pairs, 40.0).view(pairs, 2)
    u = torch.rand(3, pairs, generator=g, device=DEV, dtype=torch.float64)
    lgp = 1 + torch.sqrt(45 * ((1 + 7.43 ** 2 / 45) ** u[0] - 1))
    a = AU * (m.sum(1) * (10 ** lgp / 365.25) ** 2) ** (1 / 3)
    e = torch.sqrt(u[1])
    M = 2 * math.pi * u[2]
    E = torch.where(e < 0.8, M, torch.full_like(M, math.pi))
    for _ in range(40):
        E = E - (E - e * torch.sin(E) - M) / (1 - e * torch.cos(E))
    p = _iso(g, pairs)
    q = torch.linalg.cross(p, _iso(g, pairs))
    q = q / q.norm(dim=1, keepdim=True)
    m = m / m.sum()
    b = torch.sqrt(1 - e * e)
    w = torch.sqrt(m.sum(1) / a) / (1 - e * torch.cos(E))
    rel = (a * (torch.cos(E) - e))[:, None] * p + (a * b * torch.sin(E))[:, None] * q
    vrel = (-w * torch.sin(E))[:, None] * p + (w * b * torch.cos(E))[:, None] * q
    f = m / m.sum(1, keepdim=True)
    pos = torch.stack([cen - f[:, 1:] * rel, cen + f[:, :1] * rel], 1).view(-1, 3)
    vel = torch.stack([vel - f[:, 1:] * vrel, vel + f[:, :1] * vrel], 1).view(-1, 3)
    return pos, vel, m.reshape(-1)


def _particles(case, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    n = case["n"]
    if case["masses"] == "binaries":
        pos, vel, mass = _binaries(g, n // 2)
    else:
        pos, vel = _plummer(g, n)
        mass = torch.full((n,), 1.0 / n, device=DEV, dtype=torch.float64)
        if case["masses"] == "kroupa":
            mass = _kroupa(g, n)
            mass = mass / mass.sum()
    pos = pos - (mass[:, None] * pos).sum(0)
    vel = vel - (mass[:, None] * vel).sum(0)
    return pos.contiguous(), vel.contiguous(), mass.contiguous()


def _clusters(case, seed):
    """Independent Kroupa Plummer spheres, sizes log-uniform in [nmin, nmax] (fixed by the case, so that
    a seed changes the particles only), r_out from the first-guess recipe 0.2 n^(-1/3)."""
    r = np.random.RandomState(case["sets"] * 7919 + case["nmin"])
    sizes = np.exp(r.uniform(math.log(case["nmin"]), math.log(case["nmax"]), case["sets"])).astype(int)
    pos, _, _ = _particles({"n": int(sizes.sum()), "masses": "equal"}, seed)
    mass = _kroupa(torch.Generator(device=DEV).manual_seed(seed + 1), int(sizes.sum()))
    out, b = [], 0
    for n in map(int, sizes):
        p, m = pos[b:b + n], mass[b:b + n]
        m = (m / m.sum()).contiguous()
        out.append({"pos": (p - (m[:, None] * p).sum(0)).contiguous(), "mass": m,
                    "r_out": 0.2 * n ** (-1 / 3), "r_in": 0.02 * n ** (-1 / 3)})
        b += n
    return out


def _binary_sites(case, seed):
    """Centres of mass (at particles), measure distances, and one query offset per binary."""
    g = torch.Generator(device=DEV).manual_seed(seed + 2)
    pos, _, mass = _particles(case, seed)
    at = torch.randint(0, case["n"], (case["bins"],), generator=g, device=DEV)
    dc = torch.full((case["bins"],), 1e-3, device=DEV, dtype=torch.float64)
    return pos, mass, pos[at].contiguous(), dc, 5e-4 * _iso(g, case["bins"])


def _params(case):
    return B.Params(theta=case["theta"], r_in=0.1 * case.get("r_out", 0.05), r_out=case.get("r_out", 0.05),
                    n_leaf=case["n_leaf"], n_group=case["n_group"], order=case["order"],
                    precision=B.PT_MIXED if case["precision"] == "mixed" else B.PT_FP64,
                    mass_dependent=case.get("md", 0))


def _empty(*shape, dtype=torch.float64):
    return torch.empty(shape, dtype=dtype, device=DEV)


def _given(case, x):
    """A result in the precision it was asked in."""
    return x.float() if case["precision"] == "mixed" else x


def _orbit_dt(case):
    return 0.3 * case["r_out"] / 0.41


# ---- one pass --------------------------------------------------------------

def prepare(case, seed):
    ctx = B.Context(0)
    s = {"case": case, "ctx": ctx, "params": _params(case)}
    if case["kind"] == "batch":
        s["sets"] = _clusters(case, seed)
        n = sum(len(c["mass"]) for c in s["sets"])
        # every set's results in its slice of one array, its neighbour lists in 8 n + 64 entries of another
        s["acc"], s["pot"] = _empty(n, 3), _empty(n)
        s["nb_off"] = _empty(n + len(s["sets"]), dtype=torch.int64)
        s["nb_idx"] = torch.full((8 * n + 64 * len(s["sets"]),), -1, dtype=torch.int32, device=DEV)
        s["descs"] = (B.pt_cluster_desc * len(s["sets"]))()
        b = 0
        for k, (c, d) in enumerate(zip(s["sets"], s["descs"])):
            d.n, d.r_in, d.r_out, d.nb_capacity = len(c["mass"]), c["r_in"], c["r_out"], 8 * len(c["mass"]) + 64
            d.pos, d.mass = c["pos"].data_ptr(), c["mass"].data_ptr()
            d.acc, d.pot = s["acc"][b:].data_ptr(), s["pot"][b:].data_ptr()
            d.nb_offsets, d.nb_idx = s["nb_off"][b + k:].data_ptr(), s["nb_idx"][8 * b + 64 * k:].data_ptr()
            b += d.n
        return s
    if case["kind"] == "tidal":
        pos, mass, s["cm"], s["dc"], s["rel"] = _binary_sites(case, seed)
        bins, per = case["bins"], 1 + B.TIDAL_POINTS[case["tidal_order"]]
        # the stars, then per binary its centre and its measure points as zero-mass particles
        s["pos"] = torch.cat([pos, _empty(bins * per, 3)])
        s["points"] = s["pos"][case["n"]:].view(bins, per, 3)
        s["points"][:] = s["cm"][:, None]
        s["mass"] = torch.cat([mass, torch.zeros(bins * per, dtype=torch.float64, device=DEV)])
        s["owner"] = torch.arange(bins, device=DEV)
    else:
        s["pos"], s["vel"], s["mass"] = _particles(case, seed)
    n = s["mass"].shape[0]
    s["acc"], s["pot"] = _empty(n, 3), _empty(n)
    s["cap"] = 16 * n + 4096
    s["nb_off"] = _empty(n + 1, dtype=torch.int64)
    s["nb_idx"] = torch.full((s["cap"],), -1, dtype=torch.int32, device=DEV)
    s["tree"] = B.Tree(ctx, s["pos"], s["mass"], s["params"])
    if case["kind"] == "orbit":
        s["r_nb"] = _empty(n)
        s["orbit"] = B.pt_orbit_params(_orbit_dt(case), 3.0, 1.5, B.PT_ORBIT_ROUT)
    return s


def run(state):
    s, case = state, state["case"]
    if case["kind"] == "batch":
        rc = B.lib().pt_batch_longrange_force(s["ctx"].h, len(s["descs"]), s["descs"], s["params"].c(),
                                              B.PT_BATCH_GRAPH, None)
        s["ctx"].check(rc, "pt_batch_longrange_force")
        return {"acc": _given(case, s["acc"]), "pot": _given(case, s["pot"]), "nb_off": s["nb_off"],
                "nb_idx": s["nb_idx"]}
    tree = s["tree"]
    if case["kind"] == "orbit":
        rc, _, _ = B.pt_orbit_neighbours(tree.h, s["vel"].data_ptr(), s["orbit"], s["nb_off"].data_ptr(),
                                         s["nb_idx"].data_ptr(), s["cap"], s["r_nb"].data_ptr())
        s["ctx"].check(rc, "pt_orbit_neighbours")
        return {"nb_off": s["nb_off"], "nb_idx": s["nb_idx"], "r_nb": s["r_nb"]}
    if case["kind"] == "tidal":
        order, bins = case["tidal_order"], case["bins"]
        s["points"][:, 1:] = B.tidal_points(s["ctx"], order, s["cm"], s["dc"])
        tree.rebuild(s["pos"], s["mass"])
        tree.force(s["acc"], s["pot"])
        acc = s["acc"][case["n"]:].view(bins, -1, 3)
        T = B.tidal_tensor(s["ctx"], order, acc, s["dc"])
        at = B.tidal_eval(s["ctx"], order, s["owner"], T, acc[:, 0].contiguous(), s["rel"])
        return {"acc": s["acc"], "pot": s["pot"], "T": T, "at": at}
    tree.rebuild(s["pos"], s["mass"])
    tree.force(s["acc"], s["pot"], s["nb_off"], s["nb_idx"], s["cap"])
    return {"acc": _given(case, s["acc"]), "pot": _given(case, s["pot"]), "nb_off": s["nb_off"],
            "nb_idx": s["nb_idx"]}


# ---- what a pass cannot do without -----------------------------------------

def _interactions(n, theta):
    """Cell and particle interactions per particle of a Plummer sphere (a fit to list counts, 20%)."""
    t = (0.3 / theta) ** 2.4
    return min(n, 14000 * t / (1 + (27400 * t / n) ** 0.6))


def work(case):
    if case["kind"] == "batch":
        r = np.random.RandomState(case["sets"] * 7919 + case["nmin"])
        sizes = np.exp(r.uniform(math.log(case["nmin"]), math.log(case["nmax"]), case["sets"])).astype(int)
    else:
        per = 1 + B.TIDAL_POINTS[case["tidal_order"]] if case["kind"] == "tidal" else 0
        sizes = [case["n"] + case.get("bins", 0) * per]
    n = int(sum(sizes))
    if case["kind"] == "orbit":     # positions, masses, velocities in; lists and radii out; ~300 tests a particle
        return {"bytes": 56 * n + 8 * n + 8 * (n + 1), "flops": 10.0 * 300 * n}
    # cells (two thirds of the lists) at 55 or 22 flops each, particle pairs at 22
    each = (2 * (55 if case["order"] == 2 else 22) + 22) / 3
    flops = sum(each * m * _interactions(int(m), case["theta"]) for m in sizes)
    return {"bytes": 32 * n + 32 * n + 8 * (n + 1), "flops": float(flops)}


# ---- the same method in plain float64 --------------------------------------

def _spread(q):
    x = q & 0x1fffff
    for sh, m in ((32, 0x1f00000000ffff), (16, 0x1f0000ff0000ff), (8, 0x100f00f00f00f00f), (4, 0x10c30c30c30c30c3),
                  (2, 0x1249249249249249)):
        x = (x | (x << sh)) & m
    return x


def _expand(begin, count):
    """Concatenated ranges [begin, begin + count) and the index of the range of every entry."""
    k = torch.repeat_interleave(torch.arange(len(begin), device=DEV), count)
    off = torch.cumsum(count, 0) - count
    return begin[k] + torch.arange(len(k), device=DEV) - off[k], k


def _box(q, begin, count):
    p, k = _expand(begin, count)
    i = k[:, None].expand(-1, 3)
    lo = torch.full((len(begin), 3), 1 << 21, device=DEV).scatter_reduce(0, i, q[p], "amin")
    return lo, torch.zeros((len(begin), 3), dtype=torch.int64, device=DEV).scatter_reduce(0, i, q[p], "amax")


def _octree(x, m, key, q, n_leaf):
    """Nodes level by level: begin, count, level, leaf, first child, children, box, mass, centre, Q."""
    n = len(m)
    levels = []
    b, c = torch.zeros(1, dtype=torch.int64, device=DEV), torch.full((1,), n, device=DEV)
    for level in range(22):
        leaf = (c <= n_leaf) | torch.tensor(level == 21, device=DEV)
        p, k = _expand(b, c)
        M = torch.zeros(len(b), dtype=torch.float64, device=DEV).index_add_(0, k, m[p])
        d = x[p] - x[b][k]
        s = torch.zeros((len(b), 3), dtype=torch.float64, device=DEV).index_add_(0, k, m[p, None] * d)
        dc = torch.where(M[:, None] > 0, s / M[:, None].clamp(min=1e-300), torch.zeros_like(s))
        d = d - dc[k]
        T = torch.zeros((len(b), 3, 3), dtype=torch.float64, device=DEV)
        T.index_add_(0, k, m[p, None, None] * d[:, :, None] * d[:, None, :])
        Q = 3 * T - T.diagonal(dim1=1, dim2=2).sum(1)[:, None, None] * torch.eye(3, device=DEV, dtype=torch.float64)
        lo, hi = _box(q, b, c)
        levels.append({"b": b, "c": c, "leaf": leaf, "l": torch.full_like(b, level), "M": M, "com": x[b] + dc, "Q": Q,
                       "lo": lo, "hi": hi, "nch": torch.zeros_like(b), "fc": torch.zeros_like(b)})
        if bool(leaf.all()):
            break
        sb, sc = b[~leaf], c[~leaf]
        p, k = _expand(sb, sc)
        pre = key[p] >> (3 * (20 - level))
        new = torch.ones(len(p), dtype=torch.bool, device=DEV)
        new[1:] = (pre[1:] != pre[:-1]) | (k[1:] != k[:-1])
        at = torch.nonzero(new)[:, 0]
        b, owner = p[at], k[at]
        end = torch.cat([at[1:], torch.tensor([len(p)], device=DEV)])
        c = end - at
        nch = torch.bincount(owner, minlength=len(sb))
        levels[-1]["nch"][~leaf] = nch
        levels[-1]["fc"][~leaf] = torch.cumsum(nch, 0) - nch
    base = np.cumsum([0] + [len(v["b"]) for v in levels])
    for level, v in enumerate(levels):
        v["fc"] = v["fc"] + int(base[level + 1])
    return {k: torch.cat([v[k] for v in levels]) for k in levels[0]}


def _groups(t, n, G):
    """First particles of the walk groups."""
    b, c, leaf, fc, nch = (t[k].cpu().numpy() for k in ("b", "c", "leaf", "fc", "nch"))
    first = set()
    if c[0] <= G or leaf[0]:
        first.add(0)
    for v in np.nonzero((c > G) & ~leaf)[0]:
        cut, rb, rc = c[v] <= 8 * G, 0, 0
        for w in list(range(fc[v], fc[v] + nch[v])) + [-1]:
            if w < 0 or c[w] > G or (not cut and rc and rc + c[w] > G):
                first.update(range(rb, rb + rc, G if cut else max(rc, 1)))
                rc = 0
            if w >= 0 and c[w] > G:
                if leaf[w]:
                    first.add(int(b[w]))
            elif w >= 0:
                rb, rc = (int(b[w]) if rc == 0 else rb), rc + int(c[w])
    gb = torch.tensor(sorted(first), device=DEV)
    return gb, torch.cat([gb[1:], torch.tensor([n], device=DEV)]) - gb


def _pieces(weight, most=1 << 24):
    """Index ranges of entries whose weights sum to about `most`."""
    if not len(weight):
        return
    cum = torch.cumsum(weight, 0)
    cuts = torch.searchsorted(cum, torch.arange(most, int(cum[-1]) + most, most, device=DEV)).tolist()
    lo = 0
    for hi in cuts:
        hi = min(hi + 1, len(weight))
        if hi > lo:
            yield lo, hi
        lo = max(lo, hi)


def _tree_force(pos, mass, case, r_out):
    r_in = 0.1 * r_out
    n = len(mass)
    o = pos.amin(0)
    S = float((pos.amax(0) - o).max()) or 1.0
    scale = 2097152.0 / S
    q = torch.floor((pos - o) * scale).long().clamp(0, 2097151)
    key = (_spread(q[:, 0]) << 2) | (_spread(q[:, 1]) << 1) | _spread(q[:, 2])
    key, perm = torch.sort(key, stable=True)
    x, m, q = pos[perm], mass[perm], q[perm]
    rs = torch.ones_like(m)
    if case.get("md"):
        rs = torch.from_numpy(np.cbrt(np.maximum(1.0, (mass / mass.mean()).cpu().numpy()))).to(DEV)[perm]
    t = _octree(x, m, key, q, case["n_leaf"])
    gb, gc = _groups(t, n, case["n_group"])
    glo, ghi = _box(q, gb, gc)

    def thr(begin, count):
        p, k = _expand(begin, count)
        s = torch.zeros(len(begin), dtype=torch.float64, device=DEV).scatter_reduce(0, k, rs[p], "amax")
        return torch.floor(((r_out * s) * scale) ** 2).long() + 2

    g_thr = thr(gb, gc)
    v_thr = thr(t["b"], t["c"]) if case.get("md") else torch.zeros_like(t["b"])
    acc, phi = torch.zeros_like(x), torch.zeros_like(m)

    def cells(g, v):
        for lo, hi in _pieces(gc[g]):
            i, k = _expand(gb[g[lo:hi]], gc[g[lo:hi]])
            c = v[lo:hi][k]
            d = t["com"][c] - x[i]
            r2 = (d * d).sum(1)
            rinv = r2.rsqrt()
            mr = t["M"][c] * rinv
            f = mr / r2
            if case["order"] == 2:
                Qd = (t["Q"][c] * d[:, None, :]).sum(2)
                r5 = rinv / (r2 * r2)
                tt = (d * Qd).sum(1) * r5
                acc.index_add_(0, i, (f + 2.5 * tt / r2)[:, None] * d - Qd * r5[:, None])
                phi.index_add_(0, i, mr + 0.5 * tt)
            else:
                acc.index_add_(0, i, f[:, None] * d)
                phi.index_add_(0, i, mr)

    def pairs(g, v):
        for lo, hi in _pieces(gc[g] * t["c"][v]):
            j, k = _expand(t["b"][v[lo:hi]], t["c"][v[lo:hi]])
            gg = g[lo:hi][k]
            i, k = _expand(gb[gg], gc[gg])
            j = j[k]
            d = x[j] - x[i]
            r = torch.sqrt((d * d).sum(1))
            s = torch.maximum(rs[i], rs[j])
            u = ((r / s - r_in) / (r_out - r_in)).clamp(0, 1)
            lam = (r_out - r_in) / (r_out + r_in)
            k4 = (u - 1) ** 4 * (1 + u * (4 + u * (10 + u * (20 + u * 35 * lam))))
            w = torch.clamp(2 * r / s / (r_out + r_in) - lam * u ** 5 * (14 + u * (-28 + u * (20 - 5 * u))), max=1)
            far = (i != j) & (r > 0)
            rr = torch.where(far, r, torch.ones_like(r))
            acc.index_add_(0, i, torch.where(far, m[j] * (1 - k4) / rr ** 3, torch.zeros_like(r))[:, None] * d)
            same = torch.where(i == j, torch.zeros_like(r), 2 * m[j] / (s * (r_out + r_in)))
            phi.index_add_(0, i, torch.where(far, m[j] * w / rr, same))

    g, v = torch.arange(len(gb), device=DEV), torch.zeros(len(gb), dtype=torch.int64, device=DEV)
    theta2 = case["theta"] ** 2
    zero = torch.zeros((), dtype=torch.int64, device=DEV)
    while len(g):
        sh = 21 - t["l"][v]
        c2 = (2 * (t["lo"][v] >> sh[:, None]) + 1) << sh[:, None]
        dd = torch.maximum(torch.maximum(2 * glo[g] - c2, c2 - (2 * ghi[g] + 2)), zero)
        gap = torch.maximum(torch.maximum(t["lo"][v] - ghi[g] - 1, glo[g] - t["hi"][v] - 1), zero)
        side = (2 << sh).double()
        ok = (side * side < theta2 * (dd * dd).sum(1).double()) & ((gap * gap).sum(1) >= torch.maximum(g_thr[g], v_thr[v]))
        leaf = t["leaf"][v]
        cells(g[ok], v[ok])
        pairs(g[~ok & leaf], v[~ok & leaf])
        g, v = g[~ok & ~leaf], v[~ok & ~leaf]
        v, k = _expand(t["fc"][v], t["nch"][v])
        g = g[k]
    a, p = torch.empty_like(acc), torch.empty_like(phi)
    a[perm], p[perm] = acc, -phi
    return a, p


def exact(case, seed):
    if case["kind"] == "batch":
        sets = _clusters(case, seed)
        if sum(len(c["mass"]) for c in sets) > 600000 or len(sets) > 32:
            return None
        got = [_tree_force(c["pos"], c["mass"], case, c["r_out"]) for c in sets]
        return {"acc": torch.cat([a for a, _ in got]), "pot": torch.cat([p for _, p in got]), "nb_off": None,
                "nb_idx": None}
    if case["kind"] == "orbit":
        _, vel, mass = _particles(case, seed)
        s = torch.from_numpy(np.cbrt(np.maximum(1.0, (mass / mass.mean()).cpu().numpy()))).to(DEV) if case["md"] else 1.0
        r_nb = case["r_out"] * s + 3.0 * vel.norm(dim=1) * _orbit_dt(case)
        return {"nb_off": None, "nb_idx": None, "r_nb": r_nb}
    if case["kind"] == "tidal":
        pos, mass, cm, dc, rel = _binary_sites(case, seed)
        n, bins, h = case["n"], case["bins"], math.sqrt(0.5)
        unit = torch.tensor([[0, 0, 0], [1, 0, -h], [-1, 0, -h], [0, 1, h], [0, -1, h]], dtype=torch.float64, device=DEV)
        pts = cm[:, None] + dc[:, None, None] * unit
        a, p = _tree_force(torch.cat([pos, pts.view(-1, 3)]), torch.cat([mass, mass.new_zeros(5 * bins)]), case,
                           case["r_out"])
        meas = a[n:].view(bins, 5, 3)
        # columns xx xy xz yy yz zz of A'_i = A_ij r_j at the four unit points
        idx = [(0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2)]
        M = torch.zeros((4, 3, 6), dtype=torch.float64, device=DEV)
        for e, (i, j) in enumerate(idx):
            M[:, i, e] += unit[1:, j]
            if i != j:
                M[:, j, e] += unit[1:, i]
        T = (meas[:, 1:] - meas[:, :1]).reshape(bins, 12) @ torch.linalg.pinv(M.view(12, 6)).T / dc[:, None]
        A = T[:, [0, 1, 2, 1, 3, 4, 2, 4, 5]].view(bins, 3, 3)
        return {"acc": a, "pot": p, "T": T, "at": meas[:, 0] + (A * rel[:, None, :]).sum(2)}
    if case["n"] > 1200000:
        return None
    pos, _, mass = _particles(case, seed)
    a, p = _tree_force(pos, mass, case, case["r_out"])
    return {"acc": a, "pot": p, "nb_off": None, "nb_idx": None}
