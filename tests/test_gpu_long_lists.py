"""Groups with lists many times the mean: walked by a block and evaluated in parts.

A dense core with a sparse halo whose particles are all one walk group's (its
box spans the set, so it opens the whole tree), at set sizes around the bins
of the part length and of the block walk (2048, 8192, 32768).  Lists are sets
of the oracle's, float64 forces within 1e-10 of the oracle tree, mixed ones
within the mixed path's bound of the float64 ones (p99 1e-6), neighbours exact.
"""
import numpy as np
import pytest

import oracle
from gpu_helpers import rel_err

pytestmark = pytest.mark.gpu


def _set(n, halo, seed):
    rng = np.random.default_rng(seed)
    pos = 0.05 * rng.normal(size=(n, 3))
    pos[:halo] = 30.0 * (rng.random((halo, 3)) - 0.5)
    return pos, rng.uniform(0.5, 1.5, n) / n


@pytest.mark.parametrize("n", [2047, 2048, 8191, 8192, 32768])
@pytest.mark.parametrize("order", [0, 2])
def test_block_walk_and_parts(n, order):
    import torch

    from paper_2006_16560_gb300 import binding as B
    pos, mass = _set(n, 40, n)
    r_out = 0.02 * n ** (-1.0 / 3.0)
    T = oracle.Tree(pos, mass, 8, 64)
    a, phi, _ = T.force(0.4, 0.1 * r_out, r_out, order=order)
    off, idx = oracle.neighbours(pos, r_out)
    ctx = B.Context(0)
    dp, dm = torch.from_numpy(pos).cuda(), torch.from_numpy(mass).cuda()
    acc = torch.empty((n, 3), dtype=torch.float64, device="cuda")
    pot = torch.empty(n, dtype=torch.float64, device="cuda")
    nbo = torch.empty(n + 1, dtype=torch.int64, device="cuda")
    nbi = torch.empty(64 * n, dtype=torch.int32, device="cuda")
    for precision, p99 in ((B.PT_FP64, 1e-10), (B.PT_MIXED, 1e-6)):
        p = B.Params(theta=0.4, r_in=0.1 * r_out, r_out=r_out, n_leaf=8, n_group=64, order=order, precision=precision)
        t = B.Tree(ctx, dp, dm, p)
        prev = None
        for _ in range(3):                     # two passes, then one, then one on the replayed build
            total, st, _ = t.force(acc, pot, nbo, nbi, 64 * n)
            co, cells, po, pp = t.lists(st.cell_list_total, st.pp_list_total)
            out = [x.cpu().numpy().copy() for x in (acc, pot, nbo, nbi[:total])] + [co, cells, po, pp]
            assert prev is None or all(np.array_equal(x, y) for x, y in zip(out, prev))
            prev = out
            t.rebuild(dp, dm)
        ids = t.nodes()
        assert len(ids["begin"]) == T.nnodes
        longest = int(np.argmax(np.diff(po)))
        oc, op = T.walk(longest, 0.4, r_out)
        assert np.array_equal(np.sort(pp[po[longest]:po[longest + 1]]), np.sort(op))
        assert np.diff(co)[longest] == len(oc)
        assert np.percentile(rel_err(out[0], a), 99) <= p99
        assert np.percentile(np.abs(out[1] / phi - 1.0), 99) <= p99
        assert np.array_equal(out[2], off) and np.array_equal(out[3], idx)
        t.free()
    ctx.close()


def test_walk_stack_is_counted_per_warp():
    """max_walk_stack means pending nodes per warp whether a warp or a block walks a group:
    at most the 768 entries of a warp's stack."""
    import torch

    from paper_2006_16560_gb300 import binding as B
    pos, mass = _set(32768, 40, 1)
    ctx = B.Context(0)
    dp, dm = torch.from_numpy(pos).cuda(), torch.from_numpy(mass).cuda()
    acc = torch.empty((32768, 3), dtype=torch.float64, device="cuda")
    pot = torch.empty(32768, dtype=torch.float64, device="cuda")
    t = B.Tree(ctx, dp, dm, B.Params(theta=0.2, r_in=0.02, r_out=0.2, n_leaf=2, n_group=64, order=0,
                                     precision=B.PT_MIXED))
    for _ in range(2):
        _, st, _ = t.force(acc, pot)
        assert 32 <= st.max_walk_stack <= 768
    t.free()
    ctx.close()
