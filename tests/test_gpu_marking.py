"""Constraint marking over long columns: the walk of the changed variables'
column lists is bounded, so a system with few variables (every column in
hundreds of rows) must not spend longer on marking than on its rounds; and
results do not depend on where the bound lies."""
import time

import numpy as np
import pytest
import torch

from paper_2009_07785_gb300 import synth
from parity import compare_bounds

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def dense_columns(m, n, seed):
    """m rows of 4..12 nonzeros over n variables, a tenth of them fixed."""
    rng = np.random.default_rng(seed)
    lengths = rng.integers(4, 13, m)
    col = np.concatenate([np.sort(rng.choice(n, size=k, replace=False)) for k in lengths])
    val = np.where(rng.random(col.size) < 0.5, -1.0, 1.0) * rng.integers(1, 11, col.size)
    vt, lb, ub, x = synth._tiny_like_vars(rng, n)
    rp = synth._row_ptr(lengths)
    lhs, rhs = synth._sides(rng, rp, col, val, x, ranged_frac=0.1)
    fix = rng.random(n) < 0.1
    lb, ub = np.where(fix, x, lb), np.where(fix, x, ub)
    return synth.Instance("dense", m, n, rp, col.astype(np.int32), val, lb, ub, vt, lhs, rhs, x)


# 32 variables' lists on both sides of 512 entries, and single columns longer
# than that; up to 100k nonzeros one cluster, above the graph
@pytest.mark.parametrize("m,n", [(500, 256), (600, 256), (2000, 48), (2000, 1000), (11000, 128),
                                 (16000, 500), (16000, 8192), (16000, 9000)])
def test_long_columns_match_the_oracle(gpu, orc, m, n):
    dp, ctx = gpu
    inst = dense_columns(m, n, seed=m + n)
    d = [dev(a) for a in inst.problem()]
    with dp.Matrix(ctx, inst.m, inst.n, inst.row_ptr, inst.col, inst.val, 0, inst.lhs,
                   inst.rhs) as mat:
        a = dp.dp_propagate(ctx, mat, *d)
        b = dp.dp_propagate_hostloop(ctx, mat, *d)
    o = orc.propagate_instance(inst)
    assert a.rounds == b.rounds == o.rounds and a.infeasible == o.infeasible
    assert torch.equal(a.lb, b.lb) and torch.equal(a.ub, b.ub)
    nbad, _, det = compare_bounds(a.lb.cpu().numpy(), a.ub.cpu().numpy(), o.lb, o.ub, inst.vartype)
    assert nbad == 0, det


def test_marking_does_not_outlast_the_rounds(gpu):
    """90k nonzeros over 48 variables, a column list of 1,900 rows: one
    cluster's call against the kernels of the host-driven loop, whose marking
    ends at one changed variable.  Without a bound on the walk the call took five
    times as long as those kernels."""
    dp, ctx = gpu
    inst = dense_columns(11250, 48, seed=49)
    assert inst.nnz <= 100_000
    d = [dev(a) for a in inst.problem()]
    with dp.Matrix(ctx, inst.m, inst.n, inst.row_ptr, inst.col, inst.val, 0, inst.lhs,
                   inst.rhs) as mat:
        call, loop = [], []
        for _ in range(12):
            t0 = time.perf_counter()
            dp.dp_propagate(ctx, mat, *d)
            call.append((time.perf_counter() - t0) * 1e3)
            loop.append(sum(dp.dp_propagate_hostloop(ctx, mat, *d, timing=True).kernel_ms))
    assert min(call) < 2.5 * min(loop), (min(call), min(loop))
