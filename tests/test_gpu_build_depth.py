"""Rebuilds whose trees are deeper or shallower than the last one's.

A build launches as many levels as the tree's last build had, and a few more;
a deeper tree is noticed and built again with every level.  Each rebuild must
equal a fresh tree of the same set, whatever came before.
"""
import numpy as np
import pytest

from paper_2006_16560_gb300 import inputs

pytestmark = pytest.mark.gpu


def _sets():
    d = inputs.plummer(3000, 1)
    deep = d["pos"].copy()
    deep[1::2] = deep[::2] + 1e-7                     # tight pairs: ~20 levels with one particle per leaf
    same = d["pos"].copy()
    same[:50] = same[0]                               # coincident particles: the depth limit
    lattice = np.stack(np.meshgrid(*[np.arange(14.0)] * 3, indexing="ij"), -1).reshape(-1, 3)
    return {"plummer": d["pos"], "deep": deep, "same": same, "lattice": lattice, "two": d["pos"][:2].copy()}


@pytest.mark.parametrize("n_leaf", [1, 16])
def test_rebuild_equals_a_fresh_tree(n_leaf):
    import torch

    from paper_2006_16560_gb300 import binding as B
    ctx = B.Context(0)
    sets = {k: torch.from_numpy(np.ascontiguousarray(v)).cuda() for k, v in _sets().items()}
    p = B.Params(theta=0.5, r_in=0.002, r_out=0.02, n_leaf=n_leaf, n_group=64, order=2, precision=B.PT_MIXED)
    t = None
    for k in ("lattice", "lattice", "plummer", "plummer", "plummer", "deep", "lattice", "lattice", "same", "two", "two",
              "plummer", "same", "same", "same", "deep"):
        pos = sets[k]
        n = len(pos)
        mass = torch.full((n,), 1.0 / n, dtype=torch.float64, device="cuda")
        if t is None:
            t = B.Tree(ctx, pos, mass, p)
        else:
            t.rebuild(pos, mass)
        fresh = B.Tree(ctx, pos, mass, p)
        got, want = t.nodes(), fresh.nodes()
        for f in want:
            assert np.array_equal(got[f], want[f]), (k, f)
        assert np.array_equal(t.info()[0], fresh.info()[0])
        fresh.free()
    t.free()
    ctx.close()
