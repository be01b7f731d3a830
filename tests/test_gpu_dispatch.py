"""The rules that choose between a thread block cluster per problem (or node)
and the graph's or batched kernels: what they bound (padding, memory, the
number of problems, the size of a cluster), and that results are the same on
both sides of each."""
import time

import numpy as np
import pytest
import torch

from paper_2009_07785_gb300 import synth
from parity import compare_bounds

pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def system(lengths, n, seed, fixed=0.0):
    rng = np.random.default_rng(seed)
    lengths = np.asarray(lengths)
    col = synth._distinct_columns(rng, lengths, n)
    val = np.where(rng.random(col.size) < 0.5, -1.0, 1.0) * rng.integers(1, 11, col.size)
    vt, lb, ub, x = synth._tiny_like_vars(rng, n)
    rp = synth._row_ptr(lengths)
    lhs, rhs = synth._sides(rng, rp, col, val, x, ranged_frac=0.1)
    fix = rng.random(n) < fixed
    lb, ub = np.where(fix, x, lb), np.where(fix, x, ub)
    return synth.Instance("dispatch", lengths.size, n, rp, col, val, lb, ub, vt, lhs, rhs, x)


def check_set(dp, ctx, orc, ps, sample, slots_per_nnz):
    arrays = [dev(np.concatenate([getattr(p, a) for p in ps]))
              for a in ("lb", "ub", "vartype", "lhs", "rhs")]
    with dp.MatrixSet(ctx, ps, 0, sides=True) as ms:
        info, off = ms.info(), ms.var_off
        r = dp.dp_propagate_set(ctx, ms, *arrays)
        q = dp.dp_propagate_set_persistent(ctx, ms, *arrays)
    assert info["padded_slots"] <= slots_per_nnz * info["nnz"]
    assert np.array_equal(r.rounds, q.rounds) and np.array_equal(r.infeasible, q.infeasible)
    assert torch.equal(r.lb, q.lb) and torch.equal(r.ub, q.ub)
    for k in sample:
        p = ps[k]
        o = orc.propagate_instance(p)
        assert o.rounds == r.rounds[k] and o.infeasible == r.infeasible[k], k
        s = slice(off[k], off[k + 1])
        nbad, _, det = compare_bounds(r.lb[s].cpu().numpy(), r.ub[s].cpu().numpy(), o.lb, o.ub,
                                      p.vartype)
        assert nbad == 0, det


def test_set_of_one_row_problems_shares_slices(gpu, orc):
    """Laid out problem by problem, a row alone in its slice would take 32 slots
    to a nonzero."""
    dp, ctx = gpu
    ps = [system([40 + k % 7], 64, seed=k) for k in range(3000)]
    check_set(dp, ctx, orc, ps, range(0, 3000, 301), slots_per_nnz=1.1)


def test_set_of_many_problems_shares_slices(gpu, orc):
    """More problems than clusters run well one after the other."""
    dp, ctx = gpu
    some = [synth.tiny(seed=k, m=20, n=16) for k in range(300)]
    check_set(dp, ctx, orc, [some[k % 300] for k in range(9000)], range(0, 9000, 901),
              slots_per_nnz=1.1)


@pytest.mark.parametrize("counts", [(2, 3, 1), (24, 2)])
def test_set_of_few_rows_each(gpu, orc, counts):
    """Sets on the padded side of the rule: few slots, a cluster each."""
    dp, ctx = gpu
    rows, times = counts[:-1], counts[-1]
    ps = [synth.tiny(seed=k, m=m, n=16) for k in range(40 * times) for m in rows]
    check_set(dp, ctx, orc, ps, range(0, len(ps), 9), slots_per_nnz=24)


def test_host_nodes_are_staged_in_pieces(gpu):
    """1,200 host bound vectors of 16,000 variables, few nonzeros: 614 MB if
    staged at once.  The results are those of device-resident vectors."""
    dp, ctx = gpu
    inst = system([5] * 20, 16000, seed=4)
    LB, UB = synth.node_bounds_at_point(inst, 1200, seed=9)
    with dp.Matrix(ctx, inst.m, inst.n, inst.row_ptr, inst.col, inst.val) as mat:
        sides = [dev(a) for a in (inst.vartype, inst.lhs, inst.rhs)]
        d = dp.dp_propagate_nodes(ctx, mat, dev(LB), dev(UB), *sides)
        lb, ub = d.lb.cpu().numpy(), d.ub.cpu().numpy()
        torch.cuda.synchronize()
        free0 = torch.cuda.mem_get_info()[0]
        h = dp.dp_propagate_nodes(ctx, mat, LB, UB, inst.vartype, inst.lhs, inst.rhs)
        assert free0 - torch.cuda.mem_get_info()[0] < 300e6
        one = dp.dp_propagate_nodes(ctx, mat, LB[1100:], dev(UB[1100:]), *sides)
    assert np.array_equal(h.lb, lb) and np.array_equal(h.ub, ub)
    assert np.array_equal(h.rounds, d.rounds) and np.array_equal(h.infeasible, d.infeasible)
    assert np.array_equal(one.lb, lb[1100:]) and np.array_equal(one.rounds, d.rounds[1100:])


@pytest.mark.parametrize("lengths,count", [([5] * 64, 700), ([30, 34] * 33, 700), ([30, 34] * 33, 33)])
def test_more_nodes_than_clusters(gpu, lengths, count):
    dp, ctx = gpu
    inst = system(lengths, 96, seed=count)
    LB, UB = synth.node_bounds_at_point(inst, count, seed=2)
    args = [dev(a) for a in (LB, UB, inst.vartype, inst.lhs, inst.rhs)]
    with dp.Matrix(ctx, inst.m, inst.n, inst.row_ptr, inst.col, inst.val) as mat:
        a = dp.dp_propagate_nodes(ctx, mat, *args)
        b = dp.dp_propagate_nodes_persistent(ctx, mat, *args)
    assert np.array_equal(a.rounds, b.rounds) and np.array_equal(a.infeasible, b.infeasible)
    assert torch.equal(a.lb, b.lb) and torch.equal(a.ub, b.ub)


@pytest.mark.parametrize("lengths,n", [([200] * 100, 400), ([3] * 30000, 22500)])
def test_single_problems_by_either_path(gpu, orc, lengths, n):
    """Few long rows (a large cluster) and more slices than a cluster takes."""
    dp, ctx = gpu
    inst = system(lengths, n, seed=n, fixed=0.8 if lengths[0] > 100 else 0.0)
    assert inst.nnz <= 100_000
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


def test_cluster_is_sized_by_long_chunks(gpu):
    """100 rows of 200 nonzeros: a warp per row wants 16 blocks.  With one, as a
    warp per 32 rows would have it, the call took 2.5 times as long as the
    host-driven loop's kernels."""
    dp, ctx = gpu
    inst = system([200] * 100, 400, seed=400, fixed=0.8)
    d = [dev(a) for a in inst.problem()]
    with dp.Matrix(ctx, inst.m, inst.n, inst.row_ptr, inst.col, inst.val, 0, inst.lhs,
                   inst.rhs) as mat:
        call, loop = [], []
        for _ in range(12):
            t0 = time.perf_counter()
            dp.dp_propagate(ctx, mat, *d)
            call.append((time.perf_counter() - t0) * 1e3)
            loop.append(sum(dp.dp_propagate_hostloop(ctx, mat, *d, timing=True).kernel_ms))
    assert min(call) < 1.6 * min(loop), (min(call), min(loop))


def test_autotune_times_the_path_that_runs(gpu):
    """A problem that dp_propagate gives to a cluster is tuned by its calls: every
    entry's time is that of a call with its layout (the host-driven loop's kernels
    take up to twice as long on it)."""
    dp, ctx = gpu
    inst = synth.large(scale=0.00125)
    assert inst.nnz <= 100_000
    t = dp.dp_autotune(ctx, inst.m, inst.n, inst.row_ptr, inst.col, inst.val, inst.lb, inst.ub,
                       inst.vartype, inst.lhs, inst.rhs)
    assert {e["round_warps"] for e in t["entries"]} == {4, 8}
    assert len({e["chunk"] for e in t["entries"]}) >= 3
    d = [dev(a) for a in inst.problem()]
    for e in t["entries"]:
        with dp.Matrix(ctx, inst.m, inst.n, inst.row_ptr, inst.col, inst.val, e["chunk"], inst.lhs,
                       inst.rhs) as mat:
            best = []
            for _ in range(8):
                t0 = time.perf_counter()
                r = dp.dp_propagate(ctx, mat, *d)
                best.append((time.perf_counter() - t0) * 1e6)
        ratio = e["us_per_round"] * r.rounds / min(best)
        assert 0.6 < ratio < 1.4, (e, min(best), r.rounds)
