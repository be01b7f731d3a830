"""Propagations by one thread block cluster (a team): small single problems,
few nodes of a small matrix, sets of small problems.  The other kernels of the
library (the host-driven loop, the persistent node batch, a problem alone)
sum and screen in the same order, so results must equal theirs bit for bit,
and the oracle's within tests/parity.py's tolerance, at the sizes where the
team's code takes another path: rows of 12/13, 24/25 and 31/32/33 nonzeros,
whole rows of 256 and split ones, two-sided and one-sided slices, more
variables than are always marked one by one, a column in more rows than a
warp marks, and more items than teams."""
import numpy as np
import pytest
import torch

from paper_2009_07785_gb300 import synth
from parity import compare_bounds

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def system(lengths, n, seed, ranged=0.3, hub=False):
    rng = np.random.default_rng(seed)
    lengths = np.asarray(lengths)
    col = synth._distinct_columns(rng, lengths, n)
    rp = synth._row_ptr(lengths)
    if hub:  # column 0 in every nonempty row (the rows' smallest column)
        first = rp[:-1][lengths > 0]
        col[first] = 0
    val = np.where(rng.random(col.size) < 0.5, -1.0, 1.0) * rng.integers(1, 11, col.size)
    vt, lb, ub, x = synth._tiny_like_vars(rng, n)
    lhs, rhs = synth._sides(rng, rp, col, val, x, ranged_frac=ranged)
    return synth.Instance("team", lengths.size, n, rp, col, val, lb, ub, vt, lhs, rhs, x)


CASES = {
    "empty_and_one": lambda: system([0, 1, 0, 1, 2], 64, 1),
    "edges": lambda: system([11, 12, 13, 23, 24, 25, 31, 32, 33] * 9, 400, 2),
    "one_sided": lambda: system([3, 7, 12, 14, 24, 30] * 40, 500, 3, ranged=0.0),
    "whole_256_and_split": lambda: system([250, 255, 256, 257, 300, 513, 1100] * 3 + [5] * 200,
                                          2400, 4),
    "many_long": lambda: system([100, 200] * 120, 1200, 5),
    "marked_by_share": lambda: system(list(np.random.default_rng(6).integers(2, 9, 15000)),
                                      40000, 6, ranged=0.1),
    "hub_column": lambda: system(list(np.random.default_rng(7).integers(2, 9, 6000)), 3000, 7,
                                 hub=True),
}


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("chunk", [0, 16])
def test_team_single_equals_other_kernels(gpu, orc, name, chunk):
    dp, ctx = gpu
    inst = CASES[name]()
    assert inst.nnz <= 100_000
    d = [dev(a) for a in inst.problem()]
    with dp.Matrix(ctx, inst.m, inst.n, inst.row_ptr, inst.col, inst.val, chunk,
                   lhs=inst.lhs, rhs=inst.rhs) as mat:
        for mr in (1, 2, 100):
            p = dp.dp_params_default(max_rounds=mr)
            a = dp.dp_propagate(ctx, mat, *d, params=p)
            b = dp.dp_propagate_hostloop(ctx, mat, *d, params=p)
            assert (a.rounds, a.infeasible, a.status) == (b.rounds, b.infeasible, b.status)
            assert torch.equal(a.lb, b.lb) and torch.equal(a.ub, b.ub)
    o = orc.propagate_instance(inst)
    assert a.rounds == o.rounds and a.infeasible == o.infeasible
    nbad, _, det = compare_bounds(a.lb.cpu().numpy(), a.ub.cpu().numpy(), o.lb, o.ub, inst.vartype)
    assert nbad == 0, det


@pytest.mark.parametrize("name,count", [("edges", 1), ("edges", 130), ("edges", 700),
                                        ("whole_256_and_split", 40), ("hub_column", 9)])
@pytest.mark.parametrize("fix", [synth.node_bounds, synth.node_bounds_at_point])
def test_team_nodes_equal_the_persistent_batch(gpu, name, count, fix):
    dp, ctx = gpu
    inst = CASES[name]()
    LB, UB = fix(inst, count, seed=11)
    args = [dev(LB), dev(UB), dev(inst.vartype), dev(inst.lhs), dev(inst.rhs)]
    with dp.Matrix(ctx, inst.m, inst.n, inst.row_ptr, inst.col, inst.val) as mat:
        a = dp.dp_propagate_nodes(ctx, mat, *args)
        b = dp.dp_propagate_nodes_persistent(ctx, mat, *args)
        h = dp.dp_propagate_nodes(ctx, mat, LB, UB, inst.vartype, inst.lhs, inst.rhs)
    assert np.array_equal(a.rounds, b.rounds) and np.array_equal(a.infeasible, b.infeasible)
    assert torch.equal(a.lb, b.lb) and torch.equal(a.ub, b.ub)
    assert np.array_equal(h.lb, b.lb.cpu().numpy()) and np.array_equal(h.ub, b.ub.cpu().numpy())


@pytest.mark.parametrize("count", [1, 3, 90])
def test_team_sets_equal_the_problems_alone(gpu, count):
    dp, ctx = gpu
    names = sorted(n for n in CASES if n != "marked_by_share")
    ps = [CASES[names[k % len(names)]]() for k in range(count)]
    arrays = [dev(np.concatenate([getattr(p, a) for p in ps]))
              for a in ("lb", "ub", "vartype", "lhs", "rhs")]
    with dp.MatrixSet(ctx, ps, 0, sides=True) as ms:
        r = dp.dp_propagate_set(ctx, ms, *arrays)
        q = dp.dp_propagate_set_persistent(ctx, ms, *arrays)
        off = ms.var_off
    assert np.array_equal(r.rounds, q.rounds) and np.array_equal(r.infeasible, q.infeasible)
    assert torch.equal(r.lb, q.lb) and torch.equal(r.ub, q.ub)
    for k in range(min(count, len(names))):
        p = ps[k]
        with dp.Matrix(ctx, p.m, p.n, p.row_ptr, p.col, p.val, lhs=p.lhs, rhs=p.rhs) as mat:
            a = dp.dp_propagate(ctx, mat, *[dev(x) for x in p.problem()])
        assert a.rounds == r.rounds[k] and a.infeasible == r.infeasible[k]
        assert torch.equal(a.lb, r.lb[off[k]:off[k + 1]])
        assert torch.equal(a.ub, r.ub[off[k]:off[k + 1]])


def test_team_rejects_bad_inputs_and_survives(gpu):
    dp, ctx = gpu
    inst = CASES["edges"]()
    d = [dev(a) for a in inst.problem()]
    LB, UB = synth.node_bounds_at_point(inst, 5, seed=2)
    with dp.Matrix(ctx, inst.m, inst.n, inst.row_ptr, inst.col, inst.val) as mat:
        ref = dp.dp_propagate(ctx, mat, *d)
        nref = dp.dp_propagate_nodes(ctx, mat, dev(LB), dev(UB), *d[2:])
        for k in range(5):
            bad = [t.clone() for t in d]
            if k == 2:
                continue
            bad[k][3] = float("nan") if k != 0 else float("inf")
            with pytest.raises(dp.DomPropError) as e:
                dp.dp_propagate(ctx, mat, *bad)
            assert e.value.code == dp.DP_ERR_NAN_INPUT
            if k > 2:
                with pytest.raises(dp.DomPropError) as e:
                    dp.dp_propagate_nodes(ctx, mat, dev(LB), dev(UB), *bad[2:])
                assert e.value.code == dp.DP_ERR_NAN_INPUT
            r = dp.dp_propagate(ctx, mat, *d)
            n = dp.dp_propagate_nodes(ctx, mat, dev(LB), dev(UB), *d[2:])
            assert torch.equal(r.lb, ref.lb) and torch.equal(n.ub, nref.ub)
        keep, LB[3, 1] = LB[3, 1], np.nan
        with pytest.raises(dp.DomPropError) as e:
            dp.dp_propagate_nodes(ctx, mat, dev(LB), dev(UB), *d[2:])
        assert e.value.code == dp.DP_ERR_NAN_INPUT
        LB[3, 1] = keep
        n = dp.dp_propagate_nodes(ctx, mat, dev(LB), dev(UB), *d[2:])
        assert torch.equal(n.lb, nref.lb) and np.array_equal(n.rounds, nref.rounds)
