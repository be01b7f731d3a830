"""dp_propagate_noalloc over rows of every form its round distinguishes: rows
that one lane takes (up to 32 nonzeros), that a warp takes (up to 256; still
one FMA chain in CSR order, so the oracle's bits), and that a block takes
(longer; another order of summation, so tests/parity.py's tolerance)."""
import time

import numpy as np
import pytest
import torch

from paper_2009_07785_gb300 import synth
from parity import compare_bounds

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def system(lengths, seed):
    """Rows of the given lengths, variables and sides as the tiny workload's."""
    rng = np.random.default_rng(seed)
    lengths = np.asarray(lengths)
    n = max(64, 2 * int(lengths.max(initial=1)))
    col = synth._distinct_columns(rng, lengths, n)
    val = np.where(rng.random(col.size) < 0.5, -1.0, 1.0) * rng.integers(1, 11, col.size)
    vt, lb, ub, x = synth._tiny_like_vars(rng, n)
    rp = synth._row_ptr(lengths)
    lhs, rhs = synth._sides(rng, rp, col, val, x, ranged_frac=0.4)
    return synth.Instance("rows", lengths.size, n, rp, col, val, lb, ub, vt, lhs, rhs, x)


@pytest.mark.parametrize("lengths", [
    [0], [1], [31, 32, 33], [255, 256, 257], [0, 1, 4, 5, 32, 33, 64, 129, 256],
    [257, 300, 1023, 1024, 1025, 2049], [3] * 255 + [700], [3] * 256 + [40] * 33 + [900] * 3,
    list(range(0, 530, 7)),
])
def test_noalloc_row_forms(gpu, orc, lengths):
    dp, _ = gpu
    inst = system(lengths, seed=sum(lengths) + len(lengths))
    exact = max(lengths) <= 256
    LB, UB = synth.node_bounds_at_point(inst, 1, seed=3)
    for lb, ub in ((inst.lb, inst.ub), (LB[0], UB[0])):
        lo = torch.empty(inst.n, dtype=torch.float64, device="cuda")
        hi = torch.empty_like(lo)
        r = dp.dp_propagate_noalloc(0, torch.cuda.current_stream(), inst.m, inst.n,
                                    dev(inst.row_ptr), dev(inst.col), dev(inst.val), dev(lb),
                                    dev(ub), dev(inst.vartype), dev(inst.lhs), dev(inst.rhs), lo,
                                    hi)
        o = orc.propagate(inst.m, inst.n, inst.row_ptr, inst.col, inst.val, lb, ub, inst.vartype,
                          inst.lhs, inst.rhs)
        assert r.rounds == o.rounds and r.infeasible == o.infeasible
        lo, hi = lo.cpu().numpy(), hi.cpu().numpy()
        if exact:
            assert np.array_equal(lo, o.lb) and np.array_equal(hi, o.ub)
        else:
            nbad, _, det = compare_bounds(lo, hi, o.lb, o.ub, inst.vartype)
            assert nbad == 0, det


def call(dp, inst, lb, ub):
    lo = torch.empty(inst.n, dtype=torch.float64, device="cuda")
    hi = torch.empty_like(lo)
    args = [dev(a) for a in (inst.row_ptr, inst.col, inst.val, lb, ub, inst.vartype, inst.lhs,
                             inst.rhs)]
    return lambda: dp.dp_propagate_noalloc(0, torch.cuda.current_stream(), inst.m, inst.n, *args,
                                           lo, hi)


# rows in between whose warp takes them one by one, or a lane each; rows above
# 256 that the block takes, or a lane each; and a block of both
@pytest.mark.parametrize("lengths", [[40] * 64, [36] * 31 + [200], [33] * 20 + [1] * 12,
                                     [256, 257] * 40, [250] * 20 + [300] * 20,
                                     [20] * 31 + [3000] + [300] * 32, [0, 33] * 40])
def test_noalloc_rows_by_lane_or_together(gpu, orc, lengths):
    dp, _ = gpu
    inst = system(lengths, seed=len(lengths) + lengths[0])
    LB, UB = synth.node_bounds_at_point(inst, 1, seed=5)
    for lb, ub in ((inst.lb, inst.ub), (LB[0], UB[0])):
        r = call(dp, inst, lb, ub)()
        o = orc.propagate(inst.m, inst.n, inst.row_ptr, inst.col, inst.val, lb, ub, inst.vartype,
                          inst.lhs, inst.rhs)
        assert r.rounds == o.rounds and r.infeasible == o.infeasible
        nbad, _, det = compare_bounds(r.lb.cpu().numpy(), r.ub.cpu().numpy(), o.lb, o.ub,
                                      inst.vartype)
        assert nbad == 0, det


def test_noalloc_empty_row_out_of_its_sides(gpu):
    """A row without nonzeros has activity 0, outside [-inf, -1]."""
    dp, _ = gpu
    inst = system([0, 3, 40], seed=8)
    inst.rhs[0] = -1.0
    assert call(dp, inst, inst.lb, inst.ub)().infeasible == 1


def test_noalloc_full_warps_of_middle_rows(gpu):
    """1,000 rows of 36 nonzeros against 1,000 of 24, per round: the lanes' walks
    differ by a half.  One after the other by their warps the longer rows took
    three times as long."""
    dp, _ = gpu
    us = {}
    for k in (24, 36):
        rng = np.random.default_rng(k)
        inst = system([k] * 1000, seed=k)
        fix = rng.random(inst.n) < 0.3
        f = call(dp, inst, np.where(fix, inst.xstar, inst.lb), np.where(fix, inst.xstar, inst.ub))
        best = min(_timed(f) for _ in range(12))
        us[k] = best / f().rounds * 1e6
    assert us[36] < 2.2 * us[24], us


def _timed(f):
    t0 = time.perf_counter()
    f()
    return time.perf_counter() - t0
