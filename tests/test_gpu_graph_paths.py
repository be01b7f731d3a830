"""The captured round loops above the sizes that dp_propagate,
dp_propagate_set and dp_propagate_nodes hand to thread block clusters.  Each
input's size is checked against the dispatch limit it has to exceed: 100,000
nonzeros of a single problem or of a set's largest one, 2.5 million nonzeros
times nodes of a batch over a smaller matrix."""
import numpy as np
import pytest
import torch

from paper_2009_07785_gb300 import synth
from parity import compare_bounds

pytestmark = pytest.mark.gpu

SINGLE_NNZ = 100_000
NODE_WORK = 2_500_000


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def above(inst):
    assert inst.nnz > SINGLE_NNZ
    return inst


def mixed_lengths(m, n, seed):
    """Short rows, rows of 13..400 and a few of up to n / 3."""
    rng = np.random.default_rng(seed)
    lengths = rng.integers(1, 13, m)
    lengths[rng.random(m) < 0.03] = rng.integers(13, 401)
    lengths[rng.choice(m, 3, replace=False)] = rng.integers(n // 6, n // 3, 3)
    col = synth._distinct_columns(rng, lengths, n)
    val = np.where(rng.random(col.size) < 0.5, -1.0, 1.0) * rng.integers(1, 11, col.size)
    vt, lb, ub, x = synth._tiny_like_vars(rng, n)
    rp = synth._row_ptr(lengths)
    lhs, rhs = synth._sides(rng, rp, col, val, x, ranged_frac=0.3)
    return synth.Instance("mixed", m, n, rp, col, val, lb, ub, vt, lhs, rhs, x)


def uneven_set():
    """One problem above the limit; small ones that stop early (some infeasible), rows of every
    length, and problems without rows and with one."""
    ps = [above(mixed_lengths(14000, 12000, 5))]
    for k in range(6):
        p = synth.tiny(seed=900 + k, m=60 + 140 * k, n=50 + 100 * k)
        if k % 2:
            LB, UB = synth.node_bounds(p, 1, seed=k, lo_frac=0.05, hi_frac=0.2)
            p.lb, p.ub = LB[0], UB[0]
        ps.append(p)
    ps.append(synth.medium(seed=77, scale=0.02))
    ps.append(mixed_lengths(700, 600, 9))
    ps.append(synth.small_random(np.random.default_rng(4), 1, 12, 5))
    ps.append(synth.small_random(np.random.default_rng(6), 300, 200, 90))
    return ps


def check_problems(orc, ps, off, r, exact_rows):
    rounds = []
    for k, p in enumerate(ps):
        o = orc.propagate_instance(p)
        assert (o.rounds, o.infeasible) == (r.rounds[k], r.infeasible[k]), k
        s = slice(off[k], off[k + 1])
        lb, ub = r.lb[s].cpu().numpy(), r.ub[s].cpu().numpy()
        nbad, _, det = compare_bounds(lb, ub, o.lb, o.ub, p.vartype)
        assert nbad == 0, f"problem {k}: {det}"
        if np.diff(p.row_ptr).max() <= exact_rows:
            assert np.array_equal(lb, o.lb) and np.array_equal(ub, o.ub), k
        rounds.append(o.rounds)
    return rounds


@pytest.mark.parametrize("chunk", [0, 16])
@pytest.mark.parametrize("sides", [False, True])
def test_set_graph_loop(gpu, orc, chunk, sides):
    """Both block shapes, against the persistent loop bit for bit and every problem against
    the oracle."""
    dp, ctx = gpu
    ps = uneven_set()
    arrays = [dev(np.concatenate([getattr(p, a) for p in ps]))
              for a in ("lb", "ub", "vartype", "lhs", "rhs")]
    with dp.MatrixSet(ctx, ps, chunk, sides=sides) as ms:
        off = ms.var_off.copy()
        q = dp.dp_propagate_set_persistent(ctx, ms, *arrays)
        for warps in (8, 4):
            ms.set_launch(warps)
            r = dp.dp_propagate_set(ctx, ms, *arrays)
            assert np.array_equal(r.rounds, q.rounds) and np.array_equal(r.infeasible, q.infeasible)
            assert np.array_equal(r.cap_hit, q.cap_hit)
            assert torch.equal(r.lb, q.lb) and torch.equal(r.ub, q.ub)
        rounds = check_problems(orc, ps, off, r, chunk or 256)
        c = dp.dp_propagate_set(ctx, ms, *arrays, params=dp.dp_params_default(max_rounds=2))
    assert len(set(rounds)) > 3 and r.infeasible.any() and not r.infeasible.all()
    assert c.cap_hit.any() and c.rounds.max() == 2


def test_set_laid_out_per_problem_by_the_graph(gpu, orc):
    """A set that clusters would run, its int8 coefficients switched on: the graph's kernels
    over slices that are sorted problem by problem."""
    dp, ctx = gpu
    ps = [synth.tiny(seed=300 + k, m=40 + 90 * k, n=60 + 60 * k) for k in range(9)]
    ps.append(mixed_lengths(900, 700, 3))
    assert max(p.nnz for p in ps) <= SINGLE_NNZ
    arrays = [dev(np.concatenate([getattr(p, a) for p in ps]))
              for a in ("lb", "ub", "vartype", "lhs", "rhs")]
    with dp.MatrixSet(ctx, ps, 0, sides=True) as ms:
        off = ms.var_off.copy()
        a = dp.dp_propagate_set(ctx, ms, *arrays)
        assert ms.set_compression(True)
        for warps in (8, 4):
            ms.set_launch(warps)
            b = dp.dp_propagate_set(ctx, ms, *arrays)
            assert np.array_equal(a.rounds, b.rounds) and np.array_equal(a.infeasible, b.infeasible)
            assert torch.equal(a.lb, b.lb) and torch.equal(a.ub, b.ub)
    check_problems(orc, ps, off, b, 256)


@pytest.mark.parametrize("chunk", [0, 16])
def test_single_graph_loop_shapes_and_hostloop(gpu, orc, chunk):
    dp, ctx = gpu
    inst = above(mixed_lengths(20000, 16000, 21))
    d = [dev(a) for a in inst.problem()]
    with dp.Matrix(ctx, inst.m, inst.n, inst.row_ptr, inst.col, inst.val, chunk, inst.lhs,
                   inst.rhs) as mat:
        runs = []
        for warps in (8, 4):
            mat.set_launch(warps)
            runs.append(dp.dp_propagate(ctx, mat, *d))
            runs.append(dp.dp_propagate_hostloop(ctx, mat, *d))
        runs.append(dp.dp_propagate_persistent(ctx, mat, *d))
    a = runs[0]
    for b in runs[1:]:
        assert (a.rounds, a.infeasible, a.status) == (b.rounds, b.infeasible, b.status)
        assert torch.equal(a.lb, b.lb) and torch.equal(a.ub, b.ub)
    o = orc.propagate_instance(inst)
    assert a.rounds == o.rounds and a.infeasible == o.infeasible
    nbad, _, det = compare_bounds(a.lb.cpu().numpy(), a.ub.cpu().numpy(), o.lb, o.ub, inst.vartype)
    assert nbad == 0, det


def test_launch_shapes_of_a_small_problem(gpu):
    """Below the limit only the host-driven loop runs the kernels that the block shape
    concerns."""
    dp, ctx = gpu
    inst = synth.medium(scale=0.02)
    d = [dev(a) for a in inst.problem()]
    with dp.Matrix(ctx, inst.m, inst.n, inst.row_ptr, inst.col, inst.val, 64) as mat:
        assert mat.info()["split_rows"] > 0
        a = dp.dp_propagate_hostloop(ctx, mat, *d)
        mat.set_launch(4)
        b = dp.dp_propagate_hostloop(ctx, mat, *d)
        c = dp.dp_propagate(ctx, mat, *d)
    for x in (b, c):
        assert a.rounds == x.rounds and a.infeasible == x.infeasible
        assert torch.equal(a.lb, x.lb) and torch.equal(a.ub, x.ub)


@pytest.mark.parametrize("case,chunk,count", [("tiny", 0, 256), ("medium", 16, 200),
                                              ("medium", 0, 200)])
@pytest.mark.parametrize("fix", [synth.node_bounds, synth.node_bounds_at_point])
def test_nodes_graph_loop(gpu, orc, case, chunk, count, fix):
    dp, ctx = gpu
    inst = synth.tiny() if case == "tiny" else synth.medium(scale=0.01)
    assert inst.nnz * count > NODE_WORK
    LB, UB = fix(inst, count, seed=17)
    args = [dev(a) for a in (LB, UB, inst.vartype, inst.lhs, inst.rhs)]
    with dp.Matrix(ctx, inst.m, inst.n, inst.row_ptr, inst.col, inst.val, chunk) as mat:
        a = dp.dp_propagate_nodes(ctx, mat, *args)
        for f in (dp.dp_propagate_nodes_hostloop, dp.dp_propagate_nodes_persistent):
            b = f(ctx, mat, *args)
            assert np.array_equal(a.rounds, b.rounds) and np.array_equal(a.infeasible, b.infeasible)
            assert torch.equal(a.lb, b.lb) and torch.equal(a.ub, b.ub)
    lb, ub = a.lb.cpu().numpy(), a.ub.cpu().numpy()
    for k in range(0, count, 37):
        o = orc.propagate(inst.m, inst.n, inst.row_ptr, inst.col, inst.val, LB[k], UB[k],
                          inst.vartype, inst.lhs, inst.rhs)
        assert a.rounds[k] == o.rounds and a.infeasible[k] == o.infeasible, k
        nbad, _, det = compare_bounds(lb[k], ub[k], o.lb, o.ub, inst.vartype)
        assert nbad == 0, det


def test_batch_workspace_allocation_failures(gpu):
    """Every device allocation of a node batch's workspace fails once: the call says so, leaks
    nothing, and succeeds afterwards."""
    dp, ctx = gpu
    inst = synth.tiny()
    assert inst.nnz * 256 > NODE_WORK
    LB, UB = synth.node_bounds(inst, 256, seed=5)
    args = [dev(LB), dev(UB), dev(inst.vartype), dev(inst.lhs), dev(inst.rhs)]
    with dp.Matrix(ctx, inst.m, inst.n, inst.row_ptr, inst.col, inst.val) as ref_mat:
        ref = dp.dp_propagate_nodes(ctx, ref_mat, *args)
    with dp.Matrix(ctx, inst.m, inst.n, inst.row_ptr, inst.col, inst.val) as mat:
        live = dp.dp_debug_live_allocs()
        points = 0
        while True:
            dp.dp_debug_fail_alloc(points + 1)
            try:
                got = dp.dp_propagate_nodes(ctx, mat, *args)
                break
            except dp.DomPropError as e:
                assert e.code == dp.DP_ERR_OOM
                assert dp.dp_debug_live_allocs() == live
                points += 1
                assert points < 100
            finally:
                dp.dp_debug_fail_alloc(0)
    assert points > 15
    assert np.array_equal(got.rounds, ref.rounds) and torch.equal(got.lb, ref.lb)
