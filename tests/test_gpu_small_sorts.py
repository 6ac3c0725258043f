"""Key order and neighbour rows at the edges of the small paths.

Keys: sets at the sizes around a run (1,024), a second run and the largest
set sorted by ranks (8,192), with many equal keys (particles in few distinct
places, so that stability shows), alone and as batches of sets.  Rows: numbers
of neighbours around the per-thread (4), per-warp (32) and longest (512)
rows, and beyond it, before and after ordinary sets on the same tree.
"""
import numpy as np
import pytest

import oracle
from paper_2006_16560_gb300 import inputs

pytestmark = pytest.mark.gpu


def _cuda(x):
    import torch
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


@pytest.mark.parametrize("n", [1, 2, 3, 1000, 1023, 1024, 1025, 2048, 2049, 5000, 8191, 8192, 8193])
@pytest.mark.parametrize("places", [7, 0])
def test_key_order(n, places):
    from paper_2006_16560_gb300 import binding as B
    rng = np.random.default_rng(n + places)
    pos = rng.random((places, 3))[rng.integers(0, places, n)] if places else rng.normal(size=(n, 3))
    mass = np.full(n, 1.0 / n)
    ctx = B.Context(0)
    t = B.Tree(ctx, _cuda(pos), _cuda(mass), B.Params(n_leaf=8, n_group=64))
    keys, perm = t.keys()
    key, _, want = oracle.Tree(pos, mass, 8, 64).keys()
    assert np.array_equal(perm.astype(np.int64), want) and np.array_equal(keys, key[want])
    t.free()
    ctx.close()


@pytest.mark.parametrize("sizes", [(1, 1, 1), (700, 5, 1024, 3), (1024, 1024, 1025), (7000, 1, 1190), (7000, 1, 1191), (7000, 1, 1192)])
def test_batches_of_small_sets(sizes):
    """A batch of sets (sorted by set and key together) equals the sets alone."""
    import torch

    from paper_2006_16560_gb300 import binding as B
    ctx = B.Context(0)
    p = B.Params(theta=0.5, n_leaf=8, n_group=32, order=2, precision=B.PT_FP64)
    sets = []
    for k, n in enumerate(sizes):
        d = inputs.plummer(n, 3 + k)
        sets.append({"pos": _cuda(d["pos"]), "mass": _cuda(d["mass"]), "r_in": 0.002, "r_out": 0.02})
    b = B.Batch(sets)
    b.run(ctx, p)
    for k, st in enumerate(sets):
        q = B.Params(**{**p.__dict__, "r_in": st["r_in"], "r_out": st["r_out"]})
        acc, pot, off, idx, _ = B.longrange_force(ctx, st["pos"], st["mass"], q)
        assert torch.equal(acc, b.acc[k]) and torch.equal(pot, b.pot[k]) and torch.equal(off, b.nb_off[k])
        assert torch.equal(idx, b.nb_idx[k][: len(idx)])
    ctx.close()


def test_row_lengths():
    import torch

    from paper_2006_16560_gb300 import binding as B
    ctx = B.Context(0)
    rng = np.random.default_rng(4)
    t = None
    for clump in (2, 4, 5, 6, 33, 34, 513, 514, 6, 900, 5):       # rows of clump - 1
        pos = np.concatenate([rng.normal(size=(300, 3)), 5.0 + 1e-3 * rng.random((clump, 3)), -4.0 + 1e-3 * rng.random((7, 3))])
        n = len(pos)
        pos, mass = pos[rng.permutation(n)], np.full(n, 1.0 / n)
        p = B.Params(theta=0.5, r_in=0.001, r_out=0.01, n_leaf=8, n_group=64, order=0, precision=B.PT_MIXED)
        acc, pot = torch.empty((n, 3), dtype=torch.float64, device="cuda"), torch.empty(n, dtype=torch.float64, device="cuda")
        off, idx = torch.empty(n + 1, dtype=torch.int64, device="cuda"), torch.empty(n * n, dtype=torch.int32, device="cuda")
        dp, dm = _cuda(pos), _cuda(mass)
        if t is None:
            t = B.Tree(ctx, dp, dm, p)
        else:
            t.rebuild(dp, dm, p)
        want_off, want_idx = oracle.neighbours(pos, p.r_out)
        for _ in range(2):
            total, _, _ = t.force(acc, pot, off, idx, n * n)
            assert np.array_equal(off.cpu().numpy(), want_off)
            assert np.array_equal(idx[:total].cpu().numpy(), want_idx)
    t.free()
    ctx.close()


def test_long_rows_are_forgotten():
    """After lists with a row above 512 a tree makes short rows the short way again,
    and a tree's neighbour search along orbits does not decide for its force."""
    import torch

    from paper_2006_16560_gb300 import binding as B
    ctx = B.Context(0)
    rng = np.random.default_rng(5)
    n = 1500
    short = rng.normal(size=(n, 3))
    long = short.copy()
    long[:600] = 5.0 + 1e-3 * rng.random((600, 3))
    mass = _cuda(np.full(n, 1.0 / n))
    p = B.Params(theta=0.5, r_in=0.001, r_out=0.01, n_leaf=8, n_group=64, order=0, precision=B.PT_MIXED)
    acc, pot = torch.empty((n, 3), dtype=torch.float64, device="cuda"), torch.empty(n, dtype=torch.float64, device="cuda")
    off, idx = torch.empty(n + 1, dtype=torch.int64, device="cuda"), torch.empty(n * n, dtype=torch.int32, device="cuda")
    t = B.Tree(ctx, _cuda(short), mass, p)

    def step(pos):
        t.rebuild(_cuda(pos), mass)
        total, st, _ = t.force(acc, pot, off, idx, n * n)
        want_off, want_idx = oracle.neighbours(pos, p.r_out)
        assert np.array_equal(off.cpu().numpy(), want_off) and np.array_equal(idx[:total].cpu().numpy(), want_idx)
        return st.launches_force

    step(short)
    usual = step(short)
    assert step(long) > usual                             # made again by sorting
    assert step(long) > usual                             # by sorting at once
    step(short)
    assert step(short) == usual
    vel = _cuda(np.zeros((n, 3)))
    vel[0, 0] = 1.0
    o, i, _ = t.orbit_neighbours(vel, dt=10.0, C_v=1e9)    # one particle's radius covers the set
    assert int(np.diff(o.cpu().numpy()).max()) > 512
    assert step(short) == usual
    t.free()
    ctx.close()


def test_many_long_rows_side_by_side():
    """Clumps of adjacent particles whose rows lie around the warp's tiles (32 and 128 entries)."""
    from paper_2006_16560_gb300 import binding as B
    rng = np.random.default_rng(6)
    pos = [rng.normal(size=(500, 3))]
    for k, clump in enumerate((5, 33, 34, 64, 65, 66, 128, 129, 130, 131, 257, 258, 512, 513)):
        pos.append(np.array([10.0 + k, 0.0, 0.0]) + 1e-3 * rng.random((clump, 3)))
    pos = np.concatenate(pos)
    n = len(pos)
    ctx = B.Context(0)
    for precision in (B.PT_MIXED, B.PT_FP64):
        p = B.Params(theta=0.5, r_in=0.001, r_out=0.01, n_leaf=8, n_group=64, order=0, precision=precision)
        _, _, off, idx, _ = B.longrange_force(ctx, _cuda(pos), _cuda(np.full(n, 1.0 / n)), p, nb_capacity=n * n)
        want_off, want_idx = oracle.neighbours(pos, p.r_out)
        assert np.array_equal(off.cpu().numpy(), want_off) and np.array_equal(idx.cpu().numpy(), want_idx)
    ctx.close()
