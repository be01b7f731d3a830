"""Workloads of the propagation library as a program that uses it runs them.

A case names an entry point (`entry`), the shape of its constraint systems and
how many of them there are.  Systems are the three families of this
repository's synthetic workloads, drawn on the GPU from the seed alone:

  short      every row has 2..10 nonzeros (the tiny workload)
  mixed      97.2% rows of 2..12, 2.7% of 13..400, and one in 20,000 of
             401..100k (the large workload)
  irregular  Zipf(1.5) lengths 2..24, 30% set-partitioning rows over binaries,
             knapsack rows of up to 50k, coefficients 10^U[-2,3] (the medium
             workload)

Each is built around a feasible point, with the value, bound and variable-type
distributions of the workload of its family; matrices are loaded with the
default row split length and their sides, as a caller does that has not run
the autotuner.  Every case returns whole results: all bounds, infeasibility
flags and round counts.
"""
import math

import numpy as np
import torch

import paper_2009_07785_gb300 as dp

EPS = 1e-6        # the library's default eps_int, tau_rel and eps_feas
MAX_ROUNDS = 100  # and its default round cap


def listed():
    return [
        # one small system, device-resident: latency and launches
        {"name": "single_tiny", "entry": "single", "family": "short", "m": 2000, "n": 1500},
        # an ordinary irregular system with knapsack rows: many rounds of little work
        {"name": "single_irregular", "entry": "single", "family": "irregular", "m": 200_000,
         "n": 150_000},
        # the largest system: memory-bound rounds
        {"name": "single_large", "entry": "single", "family": "mixed", "m": 2_000_000,
         "n": 1_500_000},
        # a system whose bounds and sides live in pinned host memory, as a CPU solver's do
        {"name": "single_host", "entry": "host", "family": "mixed", "m": 400_003, "n": 300_001},
        # a dive's handful of nodes over a small matrix
        {"name": "nodes_tiny", "entry": "nodes", "family": "short", "m": 2000, "n": 1500,
         "nodes": 33, "fix": "random"},
        # strong branching: a few candidate nodes over an ordinary matrix
        {"name": "nodes_few", "entry": "nodes", "family": "irregular", "m": 200_000,
         "n": 150_000, "nodes": 8, "fix": "point"},
        # a batch of arbitrary fixings (all end infeasible after round 1: dense first rounds)
        {"name": "nodes_random", "entry": "nodes", "family": "irregular", "m": 200_000,
         "n": 150_000, "nodes": 256, "fix": "random"},
        # a batch of open nodes on the way to a solution: long runs of sparse rounds
        {"name": "nodes_point", "entry": "nodes", "family": "irregular", "m": 200_000,
         "n": 150_000, "nodes": 256, "fix": "point"},
        # a dozen small subproblems (components, cut pools) in one call
        {"name": "set_small", "entry": "set", "m_lo": 64, "m_hi": 4000, "count": 12},
        # many distinct problems of uneven size in one call
        {"name": "set_uneven", "entry": "set", "m_lo": 1000, "m_hi": 200_000, "count": 64},
        # a burst of requests to a server with resident matrices, through host memory
        {"name": "serve_burst", "entry": "serve", "m_lo": 200, "m_hi": 50_000, "count": 8,
         "requests": 256},
        # a caller that must not allocate device memory
        {"name": "noalloc", "entry": "noalloc", "family": "irregular", "m": 50_000,
         "n": 37_500},
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def mn(lo, hi):
        m = log(lo, hi)
        return {"m": m, "n": max(48, int(m * rng.uniform(0.6, 1.0)))}

    entry = rng.choice(["single", "single", "host", "nodes", "nodes", "set", "serve", "noalloc"])
    if entry in ("single", "host"):
        family = rng.choice(["short", "mixed", "irregular"])
        # irregular systems have fewer, longer rows; all stay below the largest listed case
        hi = {"short": 1_500_000, "mixed": 1_500_000, "irregular": 300_000}[family]
        return {"entry": entry, "family": family, **mn(500, hi)}
    if entry == "noalloc":
        return {"entry": entry, "family": rng.choice(["short", "irregular"]), **mn(500, 60_000)}
    if entry == "nodes":
        return {"entry": entry, "family": rng.choice(["short", "irregular"]), **mn(1000, 200_000),
                "nodes": log(1, 256), "fix": rng.choice(["random", "point"])}
    if entry == "set":
        return {"entry": entry, "m_lo": 64, "m_hi": log(500, 150_000), "count": log(2, 64)}
    return {"entry": entry, "m_lo": 200, "m_hi": log(1000, 50_000), "count": rng.randint(1, 8),
            "requests": log(1, 256)}


# ------------------------------------------------------------------ inputs --

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1_000_003 + 2009_07785) % (1 << 62))
    return g


def _uni(g, k):
    return torch.rand(k, generator=g, device="cuda", dtype=torch.float64)


def _ints(g, lo, hi, k):
    """k integers in [lo, hi)."""
    return torch.randint(lo, hi, (k,), generator=g, device="cuda", dtype=torch.int64)


def _distinct(g, rows, n):
    """A random column in [0, n) for every entry of `rows` (sorted row ids),
    distinct and ascending within each row."""
    col = _ints(g, 0, n, rows.numel())
    for _ in range(64):
        key = (rows * n + col).sort().values
        col = key - rows * n
        dup = torch.zeros(key.numel(), dtype=torch.bool, device="cuda")
        dup[1:] = key[1:] == key[:-1]
        nd = int(dup.sum())
        if nd == 0:
            return col
        col[dup] = _ints(g, 0, n, nd)
    raise RuntimeError("rows too long for their number of columns")


class System:
    """lhs <= A x <= rhs, lb <= x <= ub on the host (numpy), and a feasible point."""


def _lengths(g, family, m, n):
    if family == "short":
        return _ints(g, 2, 11, m)
    if family == "mixed":
        nlong, nmed = max(1, m // 20_000), int(0.027 * m)
        top = min(100_000, n // 2)
        ln = torch.cat([_ints(g, 2, 13, m - nmed - nlong),
                        _ints(g, 13, min(401, n // 2) + 1, nmed),
                        _ints(g, min(401, top), top + 1, nlong)])
        return ln[torch.randperm(m, generator=g, device="cuda")]
    raise ValueError(family)


def _tiny_vars(g, n):
    """60% integer (half binary, half [0, U], U in 1..20); continuous [0, U[1,100]], 10% ub = inf."""
    isint = _uni(g, n) < 0.6
    binary = isint & (_uni(g, n) < 0.5)
    ub = 1.0 + 99.0 * _uni(g, n)
    ub = torch.where(isint, _ints(g, 1, 21, n).double(), ub)
    ub = torch.where(binary, torch.ones_like(ub), ub)
    lb = torch.zeros_like(ub)
    u = _uni(g, n)
    x = torch.where(isint, torch.minimum(torch.floor(u * (ub + 1.0)), ub), u * ub)
    inf = ~isint & (_uni(g, n) < 0.1)
    ub[inf] = math.inf
    x[inf] = 100.0 * u[inf]
    return isint, lb, ub, x


def _finish(s, g, lengths, col, val, isint, lb, ub, x, ranged=None, equal=None):
    """Host arrays of the system, with sides around A x (10% ranged rows)."""
    m = lengths.numel()
    s.m, s.n = m, lb.numel()
    rp = torch.zeros(m + 1, dtype=torch.int64, device="cuda")
    rp[1:] = torch.cumsum(lengths, 0)
    s.row_ptr = rp.cpu().numpy()
    prod = (val * x[col]).cpu().numpy()
    ax = np.add.reduceat(prod, s.row_ptr[:-1])  # every row has a nonzero
    slack = -2.0 * torch.log1p(-_uni(g, 2 * m)).cpu().numpy()
    s.rhs = ax + slack[:m]
    s.lhs = np.full(m, -np.inf)
    rg = (_uni(g, m) < 0.1).cpu().numpy()
    s.lhs[rg] = ax[rg] - slack[m:][rg]
    if ranged is not None:  # rows that keep lhs = -inf
        s.lhs[ranged.cpu().numpy()] = -np.inf
    if equal is not None:   # set-partitioning rows
        e = equal.cpu().numpy()
        s.lhs[e] = s.rhs[e] = 1.0
    s.col = col.to(torch.int32).cpu().numpy()
    s.val = val.cpu().numpy()
    s.vartype = isint.to(torch.uint8).cpu().numpy()
    s.lb, s.ub, s.x = lb.cpu().numpy(), ub.cpu().numpy(), x.cpu().numpy()
    return s


def _system(family, m, n, g):
    s = System()
    if family != "irregular":
        lengths = _lengths(g, family, m, n)
        rows = torch.repeat_interleave(torch.arange(m, device="cuda"), lengths)
        col = _distinct(g, rows, n)
        nnz = col.numel()
        mag = _ints(g, 1, 11, nnz).double()
        val = torch.where(_uni(g, nnz) < 0.5, -mag, mag)
        return _finish(s, g, lengths, col, val, *_tiny_vars(g, n))
    # variables: 50% integer (half binary), 5% of the others with one infinite side
    isint = _uni(g, n) < 0.5
    binary = isint & (_uni(g, n) < 0.5)
    binary[:4] = True
    isint[:4] = True
    gen = isint & ~binary
    ub = 1.0 + 99.0 * _uni(g, n)
    ub = torch.where(gen, _ints(g, 1, 21, n).double(), ub)
    ub = torch.where(binary, torch.ones_like(ub), ub)
    lb = torch.zeros_like(ub)
    u = _uni(g, n)
    x = torch.where(isint, torch.minimum(torch.floor(u * (ub + 1.0)), ub), u * ub)
    x[binary] = (_uni(g, n) < 0.1).double()[binary]
    x[0], x[1], x[2], x[3] = 1.0, 0.0, 0.0, 0.0
    pick = ~binary & (_uni(g, n) < 0.05)
    up = _uni(g, n) < 0.5
    far = 100.0 * _uni(g, n)
    hi, lo = pick & up, pick & ~up
    x[hi] = far[hi]
    x[lo] = ub[lo] - far[lo]
    x = torch.where(isint, torch.floor(x), x)
    ub[hi] = math.inf
    lb[lo] = -math.inf
    # rows: set partitioning, others, knapsack rows
    ones = torch.nonzero(binary & (x == 1.0)).flatten()
    zeros = torch.nonzero(binary & (x == 0.0)).flatten()
    nknap = max(1, int(round(15 * m / 200_000)))
    nsp = int(0.3 * m)
    nother = m - nsp - nknap
    z = torch.arange(2, 25, device="cuda", dtype=torch.float64)
    w = z ** -1.5
    w[0] = 1.0 + w[0]                                     # Zipf(1.5), lengths 1 and 2 -> 2
    w[-1] = 2.0 / math.sqrt(23.5)                         # the tail clipped to 24
    cdf = torch.cumsum(w, 0) / w.sum()
    ln = 2 + torch.searchsorted(cdf, _uni(g, nsp + nother)).clamp(max=22)
    sp_len = torch.clamp(ln[:nsp], max=max(2, zeros.numel() // 2))
    kmax = min(50_000, max(8, n // 3))
    kmin = min(20_000, kmax)
    lengths = torch.cat([sp_len, ln[nsp:], _ints(g, kmin, kmax + 1, nknap)])
    kind = torch.cat([torch.zeros(nsp), torch.ones(nother), torch.full((nknap,), 2.0)]).cuda()
    perm = torch.randperm(m, generator=g, device="cuda")
    lengths, kind = lengths[perm], kind[perm]
    sp = kind == 0
    rows = torch.repeat_interleave(torch.arange(m, device="cuda"), lengths)
    spn = sp[rows]
    col = torch.empty(rows.numel(), dtype=torch.int64, device="cuda")
    col[~spn] = _distinct(g, rows[~spn], n)
    first = torch.zeros(rows.numel(), dtype=torch.bool, device="cuda")
    first[1:] = rows[1:] != rows[:-1]
    first[0] = True
    one, rest = spn & first, spn & ~first                 # one variable at 1, the others at 0
    col[one] = ones[_ints(g, 0, ones.numel(), int(one.sum()))]
    col[rest] = zeros[_distinct(g, rows[rest], zeros.numel())]
    key, order = (rows * n + col).sort()
    col = key - rows * n
    nnz = col.numel()
    mag = 10.0 ** (-2.0 + 5.0 * _uni(g, nnz))
    pos = (_uni(g, nnz) < 0.5) | (kind[rows] == 2)
    val = torch.where(spn, torch.ones_like(mag), torch.where(pos, mag, -mag))
    return _finish(s, g, lengths, col, val, isint, lb, ub, x, ranged=kind == 2, equal=sp)


def _node_bounds(s, count, fix, g):
    """Bound vectors that fix 1-5% of the integer variables each, to a random
    value of their domain or to the feasible point's: (lb, ub), [count, n], on the GPU."""
    lb, ub, x = (torch.from_numpy(a).cuda() for a in (s.lb, s.ub, s.x))
    ok = torch.from_numpy(s.vartype.astype(bool)).cuda() & torch.isfinite(lb) & torch.isfinite(ub)
    LB, UB = lb.repeat(count, 1), ub.repeat(count, 1)
    for b in range(count):
        share = 0.01 + 0.04 * _uni(g, 1)
        pick = torch.nonzero(ok & (_uni(g, s.n) < share)).flatten()
        if fix == "point":
            v = x[pick]
        else:
            v = lb[pick] + torch.floor(_uni(g, pick.numel()) * (ub[pick] - lb[pick] + 1.0))
        LB[b, pick] = v
        UB[b, pick] = v
    return LB, UB


def _sizes(case):
    """Row counts of a set's or a pool's systems, spread log-uniformly (by multiples of the
    golden ratio, the same for every seed)."""
    lo, hi = math.log(case["m_lo"]), math.log(case["m_hi"])
    return [int(round(math.exp(lo + (hi - lo) * ((k + 0.5) * 0.6180339887498949 % 1.0))))
            for k in range(case["count"])]


def _pool(case, g):
    """The systems of a set or pool: short and irregular in turn."""
    return [_system("short" if k % 2 == 0 else "irregular", m, max(48, 3 * m // 4), g)
            for k, m in enumerate(_sizes(case))]


def _problem(s):
    return s.lb, s.ub, s.vartype, s.lhs, s.rhs


class State:
    """What a program keeps between calls: its context, its loaded matrices, its inputs."""

    def __init__(self, entry):
        self.entry = entry
        self.ctx = dp.Context(0, torch.cuda.current_stream())
        self.mats = []
        self.server = None

    def load(self, s):
        mat = dp.Matrix(self.ctx, s.m, s.n, s.row_ptr, s.col, s.val, 0, s.lhs, s.rhs)
        self.mats.append(mat)
        return mat

    def __del__(self):
        try:
            if self.server is not None:
                self.server.close()
            for mat in self.mats:
                mat.close()
            self.ctx.close()
        except Exception:
            pass  # interpreter shutdown


def _device(arrays):
    return [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in arrays]


def prepare(case, seed):
    st = State(case["entry"])
    entry = case["entry"]
    g = _gen(seed)
    if entry in ("single", "host"):
        s = _system(case["family"], case["m"], case["n"], g)
        st.mat = st.load(s)
        if entry == "single":
            st.args = _device(_problem(s))
            st.out = (torch.empty_like(st.args[0]), torch.empty_like(st.args[0]))
        else:
            st.args = [torch.from_numpy(a).pin_memory() for a in _problem(s)]
            st.out = tuple(torch.empty(s.n, dtype=torch.float64).pin_memory() for _ in range(2))
    elif entry == "nodes":
        s = _system(case["family"], case["m"], case["n"], g)
        st.mat = st.load(s)
        st.LB, st.UB = _node_bounds(s, case["nodes"], case["fix"], g)
        st.args = _device(_problem(s)[2:])
        st.out = (torch.empty_like(st.LB), torch.empty_like(st.LB))
    elif entry == "set":
        pool = _pool(case, g)
        st.mat = dp.MatrixSet(st.ctx, pool, 0, sides=True)
        st.mats.append(st.mat)
        st.args = _device([np.concatenate([_problem(s)[k] for s in pool]) for k in range(5)])
        st.out = (torch.empty_like(st.args[0]), torch.empty_like(st.args[0]))
    elif entry == "serve":
        pool = _pool(case, g)
        st.server = dp.Server(st.ctx, slots=64)
        ids = [st.server.add_matrix(st.load(s), s.vartype, s.lhs, s.rhs) for s in pool]
        st.requests, st.lb, st.ub = [], [], []
        for k, (s, mid) in enumerate(zip(pool, ids)):
            count = _requests_of(case, k)
            LB, UB = (t.cpu().numpy() for t in _node_bounds(s, count, "point", g))
            st.lb.append(np.zeros((count, s.n)))
            st.ub.append(np.zeros((count, s.n)))
            st.requests += [(mid, LB[i], UB[i], st.lb[k][i], st.ub[k][i]) for i in range(count)]
        order = torch.randperm(len(st.requests), generator=g, device="cuda").tolist()
        st.order = order
    else:
        s = _system(case["family"], case["m"], case["n"], g)
        st.csr = _device((s.row_ptr, s.col, s.val))
        st.args = _device(_problem(s))
        st.out = (torch.empty_like(st.args[0]), torch.empty_like(st.args[0]))
        st.m, st.n = s.m, s.n
        st.stream = torch.cuda.current_stream()
    return st


def _requests_of(case, k):
    """Requests of pool matrix k: the burst dealt out evenly."""
    return case["requests"] // case["count"] + (1 if k < case["requests"] % case["count"] else 0)


# -------------------------------------------------------------------- pass --

def run(st):
    if st.entry in ("single", "host"):
        r = dp.dp_propagate(st.ctx, st.mat, *st.args, lb_out=st.out[0], ub_out=st.out[1])
    elif st.entry == "nodes":
        r = dp.dp_propagate_nodes(st.ctx, st.mat, st.LB, st.UB, *st.args, lb_out=st.out[0],
                                  ub_out=st.out[1])
    elif st.entry == "set":
        r = dp.dp_propagate_set(st.ctx, st.mat, *st.args, lb_out=st.out[0], ub_out=st.out[1])
    elif st.entry == "noalloc":
        r = dp.dp_propagate_noalloc(0, st.stream, st.m, st.n, *st.csr, *st.args, *st.out)
    else:
        return _serve(st)
    return {"lb": r.lb, "ub": r.ub, "infeasible": r.infeasible, "rounds": r.rounds}


def _serve(st):
    """The whole burst: submit every request, then poll until all are answered."""
    where, inf, rounds = {}, np.zeros(len(st.order), np.int32), np.zeros(len(st.order), np.int32)
    for i in st.order:
        mid, lb, ub, lo, hi = st.requests[i]
        where[st.server.submit(mid, lb, ub, lo, hi)] = i
    left = len(st.order)
    while left:
        for c in st.server.poll(1024, wait_us=1000):
            i = where[c["tag"]]
            inf[i], rounds[i] = c["infeasible"], c["rounds"]
            left -= 1
    return {"lb": st.lb, "ub": st.ub, "infeasible": inf, "rounds": rounds}


# -------------------------------------------------------------------- work --

def _mean_nnz(family, m, n):
    """Expected nonzeros of a system of the family."""
    if family == "short":
        return 6.0 * m
    if family == "mixed":
        nlong, nmed = max(1, m // 20_000), int(0.027 * m)
        top = min(100_000, n // 2)
        return (7.0 * (m - nmed - nlong) + 0.5 * (13 + min(400, n // 2)) * nmed +
                0.5 * (min(401, top) + top) * nlong)
    nknap = max(1, int(round(15 * m / 200_000)))
    kmax = min(50_000, max(8, n // 3))
    return 4.3 * (m - nknap) + 0.5 * (min(20_000, kmax) + kmax) * nknap


def _shapes(case):
    """(nnz, m, n, bound vectors) of the systems of one pass, expected."""
    if "family" in case:
        return [(_mean_nnz(case["family"], case["m"], case["n"]), case["m"], case["n"],
                 case.get("nodes", 1))]
    out = []
    for k, m in enumerate(_sizes(case)):
        f, n = "short" if k % 2 == 0 else "irregular", max(48, 3 * m // 4)
        vectors = _requests_of(case, k) if case["entry"] == "serve" else 1
        out.append((_mean_nnz(f, m, n), m, n, vectors))
    return out


def work(case):
    """The matrix (8-byte value, 4-byte column, 4-byte row end), sides and types
    read once, every bound vector read and written once.  Operations: one round
    over all nonzeros for every bound vector (two activity terms of a multiply
    and an add each); how many further rounds run, and over which rows, follows
    from the data."""
    by = fl = 0.0
    for nnz, m, n, vec in _shapes(case):
        by += 12.0 * nnz + 20.0 * m + n + 32.0 * n * vec
        fl += 4.0 * nnz * vec
    return {"bytes": by, "flops": fl}


def tolerance(case):
    # binary64 sums in another order.  Against exact(), whose sums run in the
    # order of its atomics, the listed and drawn cases are up to 5e-15 off; a
    # long row over small coefficients can magnify the order of its sum some
    # hundred times more.  Flags and round counts must be equal.
    return {"rel": 1e-12, "max": 1e-9}


# ------------------------------------------------------------------- exact --

def _propagate64(s, LB, UB):
    """Round-synchronous propagation of the bound vectors LB, UB ([vectors, n])
    in plain torch, binary64: (lb, ub, infeasible, rounds)."""
    dev = "cuda"
    rp = torch.from_numpy(s.row_ptr).to(dev)
    rows = torch.repeat_interleave(torch.arange(s.m, device=dev), rp[1:] - rp[:-1])
    col = torch.from_numpy(s.col).to(dev).long()
    a = torch.from_numpy(s.val).to(dev)[:, None]
    pos = a > 0
    lhs, rhs = (torch.from_numpy(v).to(dev)[:, None] for v in (s.lhs, s.rhs))
    fl, fr = torch.isfinite(lhs), torch.isfinite(rhs)
    isint = torch.from_numpy(s.vartype.astype(bool)).to(dev)[:, None]
    L, U = LB.t().contiguous().to(dev), UB.t().contiguous().to(dev)
    L, U = torch.where(isint, torch.ceil(L - EPS), L), torch.where(isint, torch.floor(U + EPS), U)
    B = L.shape[1]
    rounds = torch.zeros(B, dtype=torch.int32, device=dev)
    inf = torch.zeros(B, dtype=torch.bool, device=dev)
    alive = torch.ones(B, dtype=torch.bool, device=dev)
    intn = isint[col]
    zero = torch.zeros((), dtype=torch.float64, device=dev)

    def activity(b):
        i = torch.isinf(b)
        fin = torch.zeros(s.m, B, dtype=torch.float64, device=dev)
        fin.index_add_(0, rows, torch.where(i, zero, a * b))
        cnt = torch.zeros(s.m, B, dtype=torch.float32, device=dev)
        cnt.index_add_(0, rows, i.float())
        return fin, cnt, i

    def side(bound, b, fin, cnt, i, ok):
        """Candidates of every nonzero from one side, nan where there is none."""
        f, c = fin[rows], cnt[rows]
        res = torch.where(c == 0, f - a * b, f)
        q = (bound[rows] - res) / a
        return torch.where(ok[rows] & ((c == 0) | ((c == 1) & i)), q, torch.full_like(q, math.nan))

    def ceil_to(v, up):
        v = torch.where(intn, torch.floor(v + EPS) if up else torch.ceil(v - EPS), v)
        return torch.where(v.abs() < 1e20, v, torch.full_like(v, math.nan))

    for _ in range(MAX_ROUNDS):
        if not bool(alive.any()):
            break
        bl, bu = L[col], U[col]
        bmin, bmax = torch.where(pos, bl, bu), torch.where(pos, bu, bl)
        mn, mni, imin = activity(bmin)
        mx, mxi, imax = activity(bmax)
        bad = fr & (mni == 0) & (mn > rhs + EPS * rhs.abs().clamp(min=1.0))
        bad |= fl & (mxi == 0) & (mx < lhs - EPS * lhs.abs().clamp(min=1.0))
        r = side(rhs, bmin, mn, mni, imin, fr)
        l = side(lhs, bmax, mx, mxi, imax, fl)
        up = ceil_to(torch.where(pos, r, l), True)
        lo = ceil_to(torch.where(pos, l, r), False)
        del r, l, bmin, bmax, imin, imax
        gu = bu - torch.where(intn, zero, EPS * bu.abs().clamp(min=1.0))
        gl = bl + torch.where(intn, zero, EPS * bl.abs().clamp(min=1.0))
        up = torch.where((up < gu) | (torch.isinf(bu) & ~torch.isnan(up)), up,
                         torch.full_like(up, math.inf))
        lo = torch.where((lo > gl) | (torch.isinf(bl) & ~torch.isnan(lo)), lo,
                         torch.full_like(lo, -math.inf))
        idx = col[:, None].expand(-1, B)
        U2 = U.scatter_reduce(0, idx, up, "amin")
        L2 = L.scatter_reduce(0, idx, lo, "amax")
        del up, lo, gu, gl, bl, bu
        changed = ((U2 != U) | (L2 != L)).any(0)
        cross = torch.where(isint, L2 > U2, L2 > U2 + EPS * U2.abs().clamp(min=1.0)).any(0)
        L, U = torch.where(alive, L2, L), torch.where(alive, U2, U)
        inf |= alive & (bad.any(0) | cross)
        rounds += alive.int()
        alive &= changed & ~inf
    return L.t().contiguous(), U.t().contiguous(), inf.int(), rounds


def _in_groups(s, LB, UB, group):
    parts = [_propagate64(s, LB[b:b + group], UB[b:b + group])
             for b in range(0, LB.shape[0], group)]
    return [torch.cat([p[k] for p in parts]) for k in range(4)]


def exact(case, seed):
    entry = case["entry"]
    g = _gen(seed)
    if entry in ("single", "host", "noalloc"):
        s = _system(case["family"], case["m"], case["n"], g)
        lb, ub, inf, rounds = _propagate64(s, *(torch.from_numpy(v)[None] for v in (s.lb, s.ub)))
        return {"lb": lb[0].cpu(), "ub": ub[0].cpu(), "infeasible": int(inf[0]),
                "rounds": int(rounds[0])}
    if entry == "nodes":
        s = _system(case["family"], case["m"], case["n"], g)
        LB, UB = _node_bounds(s, case["nodes"], case["fix"], g)
        lb, ub, inf, rounds = _in_groups(s, LB, UB, 32)
        return {"lb": lb, "ub": ub, "infeasible": inf.cpu().numpy(),
                "rounds": rounds.cpu().numpy()}
    pool = _pool(case, g)
    if entry == "set":
        got = [_propagate64(s, *(torch.from_numpy(v)[None] for v in (s.lb, s.ub))) for s in pool]
        return {"lb": torch.cat([r[0][0] for r in got]), "ub": torch.cat([r[1][0] for r in got]),
                "infeasible": np.array([int(r[2][0]) for r in got], np.int32),
                "rounds": np.array([int(r[3][0]) for r in got], np.int32)}
    out = {"lb": [], "ub": [], "infeasible": [], "rounds": []}
    for k, s in enumerate(pool):
        count = _requests_of(case, k)
        LB, UB = _node_bounds(s, count, "point", g)
        if count == 0:
            for key in ("lb", "ub"):
                out[key].append(np.zeros((0, s.n)))
            continue
        lb, ub, inf, rounds = _in_groups(s, LB, UB, 32)
        for key, v in zip(("lb", "ub", "infeasible", "rounds"), (lb, ub, inf, rounds)):
            out[key].append(v.cpu().numpy())
    for key in ("infeasible", "rounds"):
        out[key] = np.concatenate(out[key]) if out[key] else np.zeros(0, np.int32)
    return out
