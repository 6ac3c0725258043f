"""Rounding errors of the float64 force kernel against float64 instructions.

The library's own tree and lists are summed on the host twice, in extended
precision (64 bits of significand or more) and in float64 as a float64 kernel
sums them (four accumulators, one list entry after another).  The kernel's
results must be no further from the extended sums than the float64 ones, in
the root mean square and at the 99th percentile of the targets.  r_out is so
small that no pair lies within it: those are float64 instructions anyway.
"""
import numpy as np
import pytest

from paper_2006_16560_gb300 import binding as B
from paper_2006_16560_gb300 import inputs

pytestmark = pytest.mark.gpu


def _sums(dtype, x, cells, parts, order):
    """Accelerations (three) and potential at x of cells (M, com, Q) and particles (m, pos)."""
    x = x.astype(dtype)
    M, com, Q = (v.astype(dtype) for v in cells)
    m, pos = (v.astype(dtype) for v in parts)
    d = com - x
    r2 = (d * d).sum(1)
    rinv = 1 / np.sqrt(r2)
    f = M * rinv * rinv * rinv
    phi = M * rinv
    a = f[:, None] * d
    if order == 2:
        qd = np.stack([Q[:, 0] * d[:, 0] + Q[:, 3] * d[:, 1] + Q[:, 4] * d[:, 2],
                       Q[:, 3] * d[:, 0] + Q[:, 1] * d[:, 1] + Q[:, 5] * d[:, 2],
                       Q[:, 4] * d[:, 0] + Q[:, 5] * d[:, 1] + Q[:, 2] * d[:, 2]], 1)
        r5 = rinv * rinv * rinv * rinv * rinv
        t = (d * qd).sum(1) * r5
        a = (f + dtype(2.5) * t * rinv * rinv)[:, None] * d - qd * r5[:, None]
        phi = phi + t / 2
    e = pos - x
    s = 1 / np.sqrt((e * e).sum(1))
    terms = np.concatenate([np.concatenate([a, (m * s * s * s)[:, None] * e]), np.concatenate([phi, m * s])[:, None]], 1)
    if dtype is np.longdouble:
        return terms.sum(0)
    # entry after entry in four accumulators (64 entries each in turn), as four warps do
    pad = np.concatenate([terms, np.zeros((-len(terms) % 256, 4))]).reshape(-1, 4, 64, 4)
    return sum(np.cumsum(pad[:, w].reshape(-1, 4), 0)[-1] for w in range(4))


def _errors(pos, mass, theta, order, n_leaf=16, targets=64, seed=0, only=None):
    import torch
    n = len(mass)
    ctx = B.Context(0)
    r_out = 1e-12 * float(np.ptp(pos, axis=0).max())
    t = B.Tree(ctx, torch.from_numpy(np.ascontiguousarray(pos)).cuda(), torch.from_numpy(mass).cuda(),
               B.Params(theta=theta, r_in=0.1 * r_out, r_out=r_out, n_leaf=n_leaf, n_group=64, order=order,
                        precision=B.PT_FP64))
    acc = torch.empty((n, 3), dtype=torch.float64, device="cuda")
    pot = torch.empty(n, dtype=torch.float64, device="cuda")
    off = torch.empty(n + 1, dtype=torch.int64, device="cuda")
    idx = torch.empty(64, dtype=torch.int32, device="cuda")
    total, st, _ = t.force(acc, pot, off, idx, 64)
    assert total == 0
    got = np.concatenate([acc.cpu().numpy(), -pot.cpu().numpy()[:, None]], 1)
    nodes, groups, (_, perm) = t.nodes(), t.groups(), t.keys()
    co, cells, po, pp = t.lists(st.cell_list_total, st.pp_list_total)
    ps, ms = pos[perm], mass[perm]
    at = np.sort(np.random.default_rng(seed).choice(n, targets, replace=False))
    if only is not None:
        at = np.nonzero(perm == only)[0]
    err = {"kernel": [], "float64": []}
    longest = 0
    for k in at:
        g = int(np.searchsorted(groups["begin"], k, side="right")) - 1
        c, p = cells[co[g]:co[g + 1]], pp[po[g]:po[g + 1]]
        p = p[p != k]
        longest = max(longest, len(c))
        lists = ((nodes["mass"][c], nodes["com"][c], nodes["quad"][c]), (ms[p], ps[p]))
        ref = _sums(np.longdouble, ps[k], *lists, order)
        for name, v in (("kernel", got[perm[k]]), ("float64", _sums(np.float64, ps[k], *lists, order))):
            d = v.astype(np.longdouble) - ref
            err[name].append((float(np.sqrt((d[:3] ** 2).sum() / (ref[:3] ** 2).sum())), float(abs(d[3] / ref[3]))))
    t.free()
    ctx.close()
    return np.array(err["kernel"]), np.array(err["float64"]), longest


def _assert_errors_no_larger(k, f):
    rms, p99 = (lambda e: np.sqrt((e * e).mean(0))), (lambda e: np.percentile(e, 99, axis=0))
    print("rms", rms(k), "float64", rms(f), "p99", p99(k), "float64", p99(f))
    assert (rms(k) <= rms(f)).all() and (p99(k) <= p99(f)).all()


def _assert_no_further(pos, mass, *args, **kw):
    k, f, longest = _errors(pos, mass, *args, **kw)
    _assert_errors_no_larger(k, f)
    return longest


@pytest.mark.parametrize("order", [0, 2])
@pytest.mark.parametrize("reach", [1e2, 1e3, 1e4, 1e5, 1e6])
def test_core_with_an_escaper(order, reach):
    """A core of unit size around the origin and one particle `reach` away, which sets the box."""
    d = inputs.plummer(3000, 5, masses="kroupa")
    pos = d["pos"].copy()
    pos[0] = [reach, 0.3 * reach, -0.1 * reach]
    _assert_no_further(pos, d["mass"], 0.4, order)


@pytest.mark.parametrize("shift", [(1e6, 0.0, 0.0), (0.0, -1e9, 1e3), (2e5, 2e5, 2e5)])
def test_sets_far_from_the_origin(shift):
    """Each axis by itself: coordinates near zero on one beside large ones on another."""
    d = inputs.plummer(2000, 6, masses="kroupa")
    _assert_no_further(d["pos"] + np.array(shift), d["mass"], 0.5, 2)


def test_flat_set():
    """A disc a millionth as thick as wide."""
    rng = np.random.default_rng(8)
    pos = rng.normal(size=(3000, 3)) * np.array([1.0, 1.0, 1e-6])
    _assert_no_further(pos, rng.uniform(0.5, 1.5, 3000) / 3000, 0.5, 2)


@pytest.mark.parametrize("theta", [0.3, 0.5, 0.6, 0.61, 0.8, 1.0, 1.5])
def test_massive_pairs_at_any_opening_angle(theta):
    """Quadrupoles that dominate: pairs of massive bodies, one cell each, and wide opening angles."""
    d = inputs.plummer(20000, 3, masses="kroupa")
    rng = np.random.default_rng(7)
    pos, mass = d["pos"].copy(), d["mass"].copy()
    for b in range(6):
        v = rng.normal(size=3)
        v *= 10.0 ** rng.uniform(-2.0, -0.3) / np.linalg.norm(v)
        c = rng.normal(size=3)
        pos[2 * b], pos[2 * b + 1] = c + v / 2, c - v / 2
        mass[2 * b] = mass[2 * b + 1] = 0.3
    _assert_no_further(pos, mass, theta, 2, targets=160)


@pytest.mark.parametrize("order", [0, 2])
def test_one_body_outweighs_a_long_list(order):
    """Thousands of cells, one of which is most of the sum: its rounding is not averaged."""
    d = inputs.plummer(60000, 4, masses="kroupa")
    pos, mass = d["pos"].copy(), d["mass"].copy()
    pos[0], mass[0] = [0.3, 0.1, -0.2], 1.0
    assert _assert_no_further(pos, mass, 0.2, order, targets=32) > 5000


def test_plummer_spheres_of_the_usual_parameters():
    for n, theta, order in ((1000, 0.5, 0), (4096, 0.5, 0), (20000, 0.3, 2), (60000, 0.6, 2)):
        d = inputs.plummer(n, n, masses="kroupa")
        _assert_no_further(d["pos"], d["mass"], theta, order, n_leaf=8)


@pytest.mark.parametrize("light", [1e-12, 1e-24, 1e-31])
def test_light_bodies_around_a_heavy_one(light):
    """The heavy body's own acceleration comes from bodies many orders lighter."""
    kernel, plain = [], []
    for body in range(17, 33):
        d = inputs.plummer(3000, 11, masses="kroupa")
        pos, mass = d["pos"].copy(), light * d["mass"]
        mass[body] = 1.0
        if body == 17:
            pos[body] = [0.01, -0.02, 0.03]
        k, f, _ = _errors(pos, mass, 0.5, 2, only=body)
        kernel.append(k[0])
        plain.append(f[0])
    _assert_errors_no_larger(np.array(kernel), np.array(plain))
