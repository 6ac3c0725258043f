"""Replayed batch graphs on inputs unlike those they were captured on.

A captured step fixes its launches and array sizes; a replay whose tree, lists
or rows do not fit must be noticed and computed again, and refused inputs must
be refused as in an uncaptured call.
"""
import numpy as np
import pytest

import oracle
from gpu_helpers import run_gpu
from paper_2006_16560_gb300 import binding as B
from paper_2006_16560_gb300 import inputs

pytestmark = pytest.mark.gpu


def _cuda(x):
    import torch
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def _batch(sizes, r_out=0.02, nb_factor=8):
    sets = []
    for k, n in enumerate(sizes):
        d = inputs.plummer(n, 40 + k, masses="kroupa")
        sets.append({"pos": _cuda(d["pos"]), "mass": _cuda(d["mass"]), "r_in": 0.1 * r_out, "r_out": r_out})
    return B.Batch(sets, nb_factor=nb_factor)


def _assert_equals_single_sets(b, prm):
    ctx = B.Context(0)
    for k, s in enumerate(b.sets):
        p = B.Params(**{**prm.__dict__, "r_in": s["r_in"], "r_out": s["r_out"]})
        g = run_gpu(ctx, s["pos"].cpu().numpy(), s["mass"].cpu().numpy(), p)
        assert np.array_equal(b.acc[k].cpu().numpy(), g["acc"]) and np.array_equal(b.pot[k].cpu().numpy(), g["pot"])
        assert np.array_equal(b.nb_off[k].cpu().numpy(), g["nb_off"])
        assert np.array_equal(b.nb_idx[k][: len(g["nb_idx"])].cpu().numpy(), g["nb_idx"])
        g["tree"].free()
    ctx.close()


@pytest.mark.parametrize("n_leaf", [1, 8])
@pytest.mark.parametrize("precision", [B.PT_FP64, B.PT_MIXED])
def test_replay_on_a_deeper_tree(n_leaf, precision):
    prm = B.Params(theta=0.5, n_leaf=n_leaf, n_group=64, order=2, precision=precision)
    ctx = B.Context(0)
    b = _batch([3000, 1500])
    for _ in range(2):
        shallow = b.run(ctx, prm, graph=True)
    pos = b.sets[0]["pos"].cpu().numpy()
    pos[:12] = pos[0] + 1e-8 * np.random.default_rng(2).random((12, 3))      # a clump far below the captured depth
    b.sets[0]["pos"].copy_(_cuda(pos))
    for _ in range(2):                                                       # the replay, and the graph captured anew
        st = b.run(ctx, prm, graph=True)
        assert st["max_level"] >= shallow["max_level"] + 5
        _assert_equals_single_sets(b, prm)
    ctx.close()


def test_replay_out_of_nodes():
    prm = B.Params(theta=0.5, n_leaf=1, n_group=64, order=2, precision=B.PT_MIXED)
    ctx = B.Context(0)
    b = _batch([3000])
    for _ in range(2):
        b.run(ctx, prm, graph=True)
    pos = b.sets[0]["pos"].cpu().numpy()
    pos[1::2] = pos[::2] + 1e-7                        # tight pairs: a chain of single children above each
    b.sets[0]["pos"].copy_(_cuda(pos))
    for _ in range(2):
        assert b.run(ctx, prm, graph=True)["nodes"] > 4 * len(pos)
        _assert_equals_single_sets(b, prm)
    ctx.close()


@pytest.mark.parametrize("what", ["nan", "inf", "negative mass"])
def test_replay_refuses_bad_input(what):
    prm = B.Params(theta=0.5, n_leaf=8, n_group=64, order=2, precision=B.PT_MIXED)
    ctx = B.Context(0)
    b = _batch([1000, 2500])
    for _ in range(2):
        b.run(ctx, prm, graph=True)
    t = b.sets[1]["mass"] if what == "negative mass" else b.sets[1]["pos"][:, 1]
    good = t[7].item()
    t[7] = {"nan": float("nan"), "inf": float("inf"), "negative mass": -good}[what]
    with pytest.raises(B.PTError) as e:
        b.run(ctx, prm, graph=True)
    assert e.value.code == B.PT_ERR_ARG
    t[7] = good
    b.run(ctx, prm, graph=True)
    _assert_equals_single_sets(b, prm)
    ctx.close()


def _clump(b, members):
    """Moves the first particles of the first set together: rows of members - 1 neighbours."""
    pos = b.sets[0]["pos"].cpu().numpy()
    pos[:members] = np.array([3.0, 1.0, 2.0]) + 1e-3 * np.random.default_rng(members).random((members, 3))
    b.sets[0]["pos"].copy_(_cuda(pos))


def _assert_rows(b):
    for k, s in enumerate(b.sets):
        off, idx = oracle.neighbours(s["pos"].cpu().numpy(), s["r_out"])
        assert np.array_equal(b.nb_off[k].cpu().numpy(), off)
        assert np.array_equal(b.nb_idx[k][: len(idx)].cpu().numpy(), idx)


def test_replay_with_rows_longer_than_captured():
    prm = B.Params(theta=0.5, n_leaf=8, n_group=64, order=0, precision=B.PT_MIXED)
    ctx = B.Context(0)
    b, other = _batch([2500, 1000], nb_factor=200), _batch([3000], nb_factor=200)
    for _ in range(2):
        b.run(ctx, prm, graph=True)
        _assert_rows(b)
    _clump(other, 700)
    other.run(ctx, prm)                                # rows too long for the captured way, in an uncaptured call
    _assert_rows(other)
    for members in (600, 40, 600, 300, 20):
        _clump(b, members)
        for _ in range(2):
            b.run(ctx, prm, graph=True)
            _assert_rows(b)
    ctx.close()


@pytest.mark.parametrize("device", [True, False])
@pytest.mark.parametrize("larger", [[9000], [300] * 40])
def test_replay_after_a_larger_batch(device, larger):
    """A batch with more particles or more sets moves the buffers that a captured one uses."""
    from test_gpu_batch import _clusters, _run_batch
    prm = B.Params(theta=0.5, n_leaf=8, n_group=64, order=2, precision=B.PT_MIXED)
    ctx = B.Context(0)
    cl = _clusters(50, [1200, 2100])
    for _ in range(2):
        rc, _, _ = _run_batch(ctx, cl, prm, flags=B.PT_BATCH_GRAPH, device=device)
        assert rc == B.PT_OK
    assert _run_batch(ctx, _clusters(60, larger), prm, device=device)[0] == B.PT_OK
    rng = np.random.default_rng(3)
    for _ in range(3):
        for c in cl:
            c["pos"] = c["pos"] + 1e-3 * rng.normal(size=c["pos"].shape)
        rc, got, _ = _run_batch(ctx, cl, prm, flags=B.PT_BATCH_GRAPH, device=device)
        assert rc == B.PT_OK
        for c, r in zip(cl, got):
            p = B.Params(**{**prm.__dict__, "r_in": c["r_in"], "r_out": c["r_out"]})
            g = run_gpu(ctx, c["pos"], c["mass"], p)
            for k in ("acc", "pot", "nb_off", "nb_idx"):
                assert np.array_equal(r[k], g[k]), k
            g["tree"].free()
    ctx.close()
