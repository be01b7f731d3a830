"""Batches of few nodes: the activity kernel that packs several chunks into a
warp (at most 16 nodes) against the one that takes a chunk per warp."""
import numpy as np
import pytest
import torch

from paper_2009_07785_gb300 import synth
from parity import compare_bounds

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def call(f, ctx, mat, inst, LB, UB):
    r = f(ctx, mat, dev(LB), dev(UB), dev(inst.vartype), dev(inst.lhs), dev(inst.rhs))
    return r.lb.cpu().numpy(), r.ub.cpu().numpy(), r.rounds, r.infeasible


# one octet of nodes and two, full and not, and the first batch above the rule
@pytest.mark.parametrize("count", [1, 7, 8, 9, 16, 17])
@pytest.mark.parametrize("chunk", [16, 256])  # split rows, whole rows
def test_few_nodes_equal_the_chunk_per_warp_kernel(gpu, orc, count, chunk):
    """The rounds of the persistent loop take a chunk per warp at every count:
    the results are the same bits, and the oracle's within rounding."""
    dp, ctx = gpu
    inst = synth.small_random(np.random.default_rng(11), 400, 300, 60)
    LB, UB = synth.node_bounds_at_point(inst, count, seed=7)
    with dp.Matrix(ctx, inst.m, inst.n, inst.row_ptr, inst.col, inst.val, chunk) as mat:
        assert (mat.info()["split_rows"] > 0) == (chunk == 16)
        a = call(dp.dp_propagate_nodes_hostloop, ctx, mat, inst, LB, UB)
        b = call(dp.dp_propagate_nodes_persistent, ctx, mat, inst, LB, UB)
    for x, y in zip(a, b):
        assert np.array_equal(x, y)
    for k in range(count):
        o = orc.propagate(inst.m, inst.n, inst.row_ptr, inst.col, inst.val, LB[k], UB[k],
                          inst.vartype, inst.lhs, inst.rhs)
        assert a[2][k] == o.rounds and a[3][k] == o.infeasible, k
        nbad, _, det = compare_bounds(a[0][k], a[1][k], o.lb, o.ub, inst.vartype)
        assert nbad == 0, det


def test_few_and_many_nodes_share_a_workspace(gpu):
    """Calls of 16, 40 and 16 nodes over one matrix that is too large for the
    team path, so that both round graphs run, on one workspace: a node's
    result does not depend on the batch it is in."""
    dp, ctx = gpu
    inst = synth.medium(scale=0.2)
    LB, UB = synth.node_bounds_at_point(inst, 40, seed=3)
    with dp.Matrix(ctx, inst.m, inst.n, inst.row_ptr, inst.col, inst.val, 64) as mat:
        assert mat.info()["nnz"] > 300_000 and mat.info()["split_rows"] > 0
        few = call(dp.dp_propagate_nodes, ctx, mat, inst, LB[:16], UB[:16])
        many = call(dp.dp_propagate_nodes, ctx, mat, inst, LB, UB)
        again = call(dp.dp_propagate_nodes, ctx, mat, inst, LB[:16], UB[:16])
    for x, y, z in zip(few, many, again):
        assert np.array_equal(x, y[:16]) and np.array_equal(x, z)


def uneven(rows, seed):
    rng = np.random.default_rng(seed)
    lengths = np.where(rng.random(rows) < 0.02, rng.integers(40, 200, rows),
                       rng.integers(1, 9, rows))
    n = 12000
    col = synth._distinct_columns(rng, lengths, n)
    val = np.where(rng.random(col.size) < 0.5, -1.0, 1.0) * rng.integers(1, 11, col.size)
    vt, lb, ub, x = synth._tiny_like_vars(rng, n)
    rp = synth._row_ptr(lengths)
    lhs, rhs = synth._sides(rng, rp, col, val, x)
    return synth.Instance("few", rows, n, rp, col, val, lb, ub, vt, lhs, rhs, x)


# more work items than warps of the activity kernel (3,648), in rows of uneven length with
# split ones among them: up to 8 nodes a step packs four chunks, up to 16 two, and
# above the items go out in fixed shares or by ticket (the persistent loop's from
# 250,000 items on)
@pytest.mark.parametrize("rows,chunk,count",
                         [(r, c, k) for r, c in ((17001, 256), (17001, 64), (9001, 16))
                          for k in (1, 7, 8, 16, 17, 40)] + [(17001, 64, 480)])
def test_batches_with_more_chunks_than_warps(gpu, orc, count, rows, chunk):
    dp, ctx = gpu
    inst = uneven(rows, seed=rows + count)
    LB, UB = synth.node_bounds_at_point(inst, count, seed=7)
    with dp.Matrix(ctx, inst.m, inst.n, inst.row_ptr, inst.col, inst.val, chunk) as mat:
        a = call(dp.dp_propagate_nodes_hostloop, ctx, mat, inst, LB, UB)
        b = call(dp.dp_propagate_nodes_persistent, ctx, mat, inst, LB, UB)
        c = call(dp.dp_propagate_nodes, ctx, mat, inst, LB, UB)
    for x, y, z in zip(a, b, c):
        assert np.array_equal(x, y) and np.array_equal(x, z)
    for k in {0, count - 1}:
        o = orc.propagate(inst.m, inst.n, inst.row_ptr, inst.col, inst.val, LB[k], UB[k],
                          inst.vartype, inst.lhs, inst.rhs)
        assert a[2][k] == o.rounds and a[3][k] == o.infeasible, k
        nbad, _, det = compare_bounds(a[0][k], a[1][k], o.lb, o.ub, inst.vartype)
        assert nbad == 0, det
