"""The float64 force kernel's float32 expansions: units, offsets and list edges.

Lengths and masses are scaled inside the kernel by powers of two, so a set
whose lengths are multiplied by 2^k and masses by 2^j must give exactly
2^(j - 2k) times the accelerations and 2^(j - k) times the potentials; and
sets far from the origin or with lists around the kernel's tile (32), fold
(64) and pass (32, 64) sizes must match the oracle's tree to the float64
bound of the other parity tests (1e-10).
"""
import numpy as np
import pytest

import oracle
from gpu_helpers import rel_err
from paper_2006_16560_gb300 import inputs

pytestmark = pytest.mark.gpu


def _run(pos, mass, **kw):
    import torch

    from paper_2006_16560_gb300 import binding as B
    ctx = B.Context(0)
    acc, pot, off, idx, _ = B.longrange_force(ctx, torch.from_numpy(pos).cuda(), torch.from_numpy(mass).cuda(),
                                              B.Params(precision=B.PT_FP64, **kw))
    out = acc.cpu().numpy(), pot.cpu().numpy(), off.cpu().numpy(), idx.cpu().numpy()
    ctx.close()
    return out


@pytest.mark.parametrize("k,j", [(-300, 7), (-40, -90), (40, 0), (100, 300)])
def test_power_of_two_units(k, j):
    d = inputs.plummer(3001, 5, masses="kroupa")
    kw = dict(theta=0.5, n_leaf=8, n_group=64, order=2)
    a0, p0, o0, i0 = _run(d["pos"], d["mass"], r_in=0.003, r_out=0.03, **kw)
    s, m = 2.0 ** k, 2.0 ** j
    a, p, o, i = _run(d["pos"] * s, d["mass"] * m, r_in=0.003 * s, r_out=0.03 * s, **kw)
    assert np.array_equal(o, o0) and np.array_equal(i, i0)
    # every step is exactly scale free; two factors, so that neither leaves float64's range
    assert np.array_equal(a, a0 * 2.0 ** (j - k) * 2.0 ** -k)
    assert np.array_equal(p, p0 * 2.0 ** (j - k))


@pytest.mark.parametrize("shift", [1.0e3, 1.0e4])
def test_sets_far_from_the_origin(shift):
    d = inputs.plummer(2000, 6, masses="kroupa")
    pos = d["pos"] + np.array([shift, -2.0 * shift, 0.25 * shift])
    a, p, off, idx = _run(pos, d["mass"], theta=0.4, r_in=0.004, r_out=0.04, n_leaf=8, n_group=64, order=2)
    T = oracle.Tree(pos, d["mass"], 8, 64)
    ao, po, _ = T.force(0.4, 0.004, 0.04, order=2)
    assert rel_err(a, ao).max() <= 1e-10
    np.testing.assert_allclose(p, po, rtol=1e-10)
    assert np.array_equal(off, oracle.neighbours(pos, 0.04)[0])


@pytest.mark.parametrize("n", [2, 3, 31, 32, 33, 63, 64, 65, 129, 257])
@pytest.mark.parametrize("r_out", [1e-6, 0.1, 3.0])
def test_list_and_pass_edges(n, r_out):
    """theta = 0 puts every particle in every list: lengths at the edges of
    tiles, folds and passes, with no, some and all pairs within r_out."""
    d = inputs.plummer(n, 9, masses="kroupa")
    for n_group in (32, 128):
        a, p, off, idx = _run(d["pos"], d["mass"], theta=0.0, r_in=0.1 * r_out, r_out=r_out, n_leaf=4,
                              n_group=n_group, order=2)
        ao, po = oracle.direct_force(d["pos"], d["mass"], 0.1 * r_out, r_out)
        assert np.abs(a - ao).max() <= 1e-10 * np.abs(ao).max()
        np.testing.assert_allclose(p, po, rtol=1e-10)
        oo, oi = oracle.neighbours(d["pos"], r_out)
        assert np.array_equal(off, oo) and np.array_equal(idx, oi)


@pytest.mark.parametrize("k,j", [(400, -300), (480, -100), (320, -760)])
def test_units_below_the_smallest_number(k, j):
    """Units in which accelerations or potentials fall below float64's range: zero, not
    infinity times zero (near pairs are scaled by 1 / unit)."""
    d = inputs.plummer(500, 5, masses="kroupa")
    kw = dict(theta=0.5, n_leaf=8, n_group=64, order=2)
    _, p0, o0, i0 = _run(d["pos"], d["mass"], r_in=0.05, r_out=0.5, **kw)
    s = 2.0 ** k
    a, p, o, i = _run(d["pos"] * s, d["mass"] * 2.0 ** j, r_in=0.05 * s, r_out=0.5 * s, **kw)
    assert len(i0) > 500 and np.array_equal(o, o0) and np.array_equal(i, i0)
    assert np.isfinite(a).all() and np.isfinite(p).all()
    assert np.abs(a).max() <= 1e-300
    if k - j < 1000:
        assert np.array_equal(p, p0 * 2.0 ** (j - k))
    else:
        assert np.abs(p).max() <= 1e-300


@pytest.mark.parametrize("k,j", [(20, -950), (-30, -1005), (0, -1010)])
def test_units_near_the_smallest_number(k, j):
    """Accelerations and potentials just above float64's smallest normal number, near pairs among them."""
    d = inputs.plummer(500, 5, masses="kroupa")
    mass = np.ldexp(np.rint(np.ldexp(d["mass"], 24)), -24)      # few bits: exact in any unit
    kw = dict(theta=0.0, n_leaf=8, n_group=64, order=0)
    a0, p0, o0, i0 = _run(d["pos"], mass, r_in=0.05, r_out=0.5, **kw)
    s = 2.0 ** k
    a, p, o, i = _run(d["pos"] * s, mass * 2.0 ** j, r_in=0.05 * s, r_out=0.5 * s, **kw)
    assert len(i0) > 500 and np.array_equal(o, o0) and np.array_equal(i, i0)
    # near pairs lose bits where m / r^3 falls below the smallest normal number
    assert np.abs(a * 2.0 ** 900 * 2.0 ** (2 * k - j - 900) - a0).max() <= 1e-10 * np.abs(a0).max()
    assert np.abs(p * 2.0 ** 900 * 2.0 ** (k - j - 900) - p0).max() <= 1e-10 * np.abs(p0).max()
