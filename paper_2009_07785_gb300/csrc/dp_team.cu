// Whole propagations by a team of blocks (Alg. 2 of arXiv 2009.07785, every
// round of it, its prologue and its epilogue in one launch).  A team is a
// thread block cluster; the teams of a launch take one small problem each and
// share nothing but the matrix.
//
// What bounds the propagation of a small problem is not bytes but the chain
// of dependent steps of a round and the number of rounds (20 to 30).  So here
//   - rounds are separated by cluster barriers (0.2-0.3 us for 16 blocks)
//     instead of three to five kernels;
//   - from the second round on only the chunks are processed that hold a
//     variable that changed in the round before (the constraint marking of
//     Alg. 1, Sec. 2.1), found through the columns of the changed variables.
//     Skipping the others is exact: their activities, hence their candidates,
//     are those of the round that processed them last, applied or rejected
//     then against bounds that have only tightened since;
//   - surviving nonzeros wait in a per-warp buffer and are evaluated 32 at a
//     time (the binary64 pipe takes 64 clocks per warp instruction, however
//     many lanes are active), without a queue in memory or a phase of their
//     own: the records they read do not change before the round's commit.
// The arithmetic is that of dp_kernels.cu and dp_batch.cu: one FMA chain per
// chunk in CSR order, the same association of split rows' pieces, the same
// screen and candidates, so results are the same bits.
#include <cuda_runtime.h>
#include <cstdint>
#include <cfloat>

#include "dp_device.cuh"
#include "dp_internal.h"
#include "dp_launch.h"
#include "dp_round.cuh"
#include "../../include/domprop.h"

namespace dp {

namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kPairCap = 64;

// Nonzeros that survived the screen, with their rows' sums (warp-private).
struct Pairs {
  uint32_t off[kPairCap];   // element offset in val/col
  uint32_t cs[kPairCap];    // chunk slot << 2 | sides
  double minfin[kPairCap], maxfin[kPairCap];
  uint32_t ninf[kPairCap];  // bit 0: mininf == 0, bit 1: maxinf == 0
};

// One team's view of the arrays (its slot of the state), one copy per block
// in shared memory: kept in registers it would cost the phases theirs.  For
// the same reason the phases are functions of their own.
struct Team {
  VarRec *rec;
  longlong2 *keys;
  uint32_t *dirty, *mask;
  int32_t *touch;
  Partial *part;
  RowTot *rowtot;
  TeamFlags *flags;
  TeamView v;
  int nw;        // the team's warps
  int rank, nb;  // this block among the team's blocks
  int round, p;  // executed rounds, and their parity
  int64_t nmask; // slices: round r reads masks p * nmask + slice and marks in the others
  // this warp among the team's: consecutive ones on different blocks, since
  // slices are sorted by length
  __device__ __forceinline__ int gw() const { return (int)(threadIdx.x >> 5) * nb + rank; }
};

__device__ __forceinline__ void ld_rec_l2(const VarRec *q, double &L, double &U, float &WU,
                                          float &WL, uint32_t &flags) {
  double d2, d3;
  asm volatile("ld.global.cg.v4.f64 {%0,%1,%2,%3}, [%4];"
               : "=d"(L), "=d"(U), "=d"(d2), "=d"(d3)
               : "l"(q));
  const long long w = __double_as_longlong(d2);
  WU = __int_as_float((int)(w & 0xFFFFFFFFll));
  WL = __int_as_float((int)((unsigned long long)w >> 32));
  flags = (uint32_t)((unsigned long long)__double_as_longlong(d3) & 0xFFFFFFFFull);
}

// Writes a variable's record.
__device__ __forceinline__ void put_var(VarRec *q, double L, double U, bool isint, float tau_dn,
                                        float eps_dn) {
  float WU, WL;
  screen_widths(L, U, isint, tau_dn, eps_dn, WU, WL);
  reinterpret_cast<double2 *>(q)[0] = make_double2(L, U);
  reinterpret_cast<uint4 *>(q)[1] =
      make_uint4(__float_as_uint(WU), __float_as_uint(WL), isint ? 1u : 0u, 0u);
}

// ------------------------------------------------------------- barriers --

__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release;\n"
               "barrier.cluster.wait.acquire;" ::
                   : "memory");
}

// ----------------------------------------------------------- candidates --

// Evaluates buffered pairs [from, from + count), count <= 32: the candidates
// of one nonzero per lane, applied to the next state with order-preserving
// 64-bit atomics that nothing waits for; the changed variables are marked in
// the dirty bitmap.  All 32 lanes call.
__device__ __noinline__ void eval_pairs(const TeamArgs &A, const Team &T, const Pairs &B,
                                           int from, int count) {
  __syncwarp();
  const int lane = threadIdx.x & 31;
  if (lane < count) {
    const int q = from + lane;
    const uint32_t off = B.off[q], cs = B.cs[q], ninf = B.ninf[q];
    const double a = __ldg(A.M.val + off);
    const int32_t j = __ldg(A.M.col + off);
    const double2 sd = __ldcg(A.side + (cs >> 2));
    double L, U;
    float WU, WL;
    uint32_t fl;
    ld_rec_l2(T.rec + j, L, U, WU, WL, fl);
    RowView rv;
    rv.minfin = B.minfin[q];
    rv.maxfin = B.maxfin[q];
    rv.mininf = (ninf & 1u) ? 0 : 1;
    rv.maxinf = (ninf & 2u) ? 0 : 1;
    rv.lhs = sd.x;
    rv.rhs = sd.y;
    const bool isint = (fl & 1u) != 0u;
    const unsigned sides = cs & 3u;
    bool any = false;
    auto apply = [&](const SideCand &c) {
      if (!c.apply) return;
      if (c.upper) atomicMin(&T.keys[j].y, key_of(c.v));
      else atomicMax(&T.keys[j].x, key_of(c.v));
      any = true;
    };
    apply(side_candidate(a, L, U, isint, (sides & 1u) != 0u, rv, A.eps_int, A.tau_rel,
                         A.inf_thr));
    if (sides == 3u)
      apply(side_candidate(a, L, U, isint, false, rv, A.eps_int, A.tau_rel, A.inf_thr));
    if (any) {
      const int32_t b = j - T.v.var0;
      atomicOr(&T.dirty[T.v.dword0 + (b >> 5)], 1u << (b & 31));
      T.flags->changed[T.p] = 1;
    }
  }
  __syncwarp();
}

// Buffers the nonzero `off` of every lane with h set and evaluates 32 pairs
// as soon as there are that many.  n: buffered pairs (warp-uniform).
__device__ __forceinline__ void push_pair(bool h, const TeamArgs &A, const Team &T, Pairs &B,
                                          int &n, int64_t off, int64_t slot, unsigned sides,
                                          const RowView &rv) {
  const unsigned m = __ballot_sync(kFull, h);
  if (m == 0u) return;
  if (h) {
    const int q = n + __popc(m & ((1u << (threadIdx.x & 31)) - 1u));
    B.off[q] = (uint32_t)off;
    B.cs[q] = ((uint32_t)slot << 2) | sides;
    B.minfin[q] = rv.minfin;
    B.maxfin[q] = rv.maxfin;
    B.ninf[q] = (rv.mininf == 0 ? 1u : 0u) | (rv.maxinf == 0 ? 2u : 0u);
  }
  n += __popc(m);
  if (n >= 32) {
    n -= 32;
    eval_pairs(A, T, B, n, 32);
  }
}

// Survivors that can be named without a re-read (as enqueue_named of the
// graph's kernels): with one screen value of a side above the threshold only
// the chunk's largest, with one infinite contribution only that nonzero.
// Returns whether the lane's chunk needs the re-read.  All 32 lanes call.
__device__ __forceinline__ bool push_named(const TeamArgs &A, const Team &T, Pairs &B, int &n,
                                           const RowView &rv, const Top2 &t, int chunk_mininf,
                                           int chunk_maxinf, int64_t slot, int64_t elem0) {
  const bool act = rv.act != 0;
  if (__ballot_sync(kFull, act) == 0u) return false;
  const bool full = act && (rv.exact || (rv.mininf == 0 && t.r2 > rv.thr_r) ||
                            (rv.maxinf == 0 && t.l2 > rv.thr_l));
  bool h1 = false, h2 = false;
  int k1 = 0, k2 = 0;
  if (act && !full) {
    const bool fr = d_isfinite(rv.rhs), fl = d_isfinite(rv.lhs);
    if (fr && rv.mininf == 0 && t.r1 > rv.thr_r) { h1 = true; k1 = t.kr; }
    if (fr && rv.mininf == 1 && chunk_mininf > 0) { h1 = true; k1 = t.kinf_min; }
    if (fl && rv.maxinf == 0 && t.l1 > rv.thr_l) { h2 = true; k2 = t.kl; }
    if (fl && rv.maxinf == 1 && chunk_maxinf > 0) { h2 = true; k2 = t.kinf_max; }
  }
  const bool both = h1 && h2 && k1 == k2;
  push_pair(h1, A, T, B, n, elem0 + (int64_t)k1 * kSliceW, slot, both ? 3u : 1u, rv);
  push_pair(h2 && !both, A, T, B, n, elem0 + (int64_t)k2 * kSliceW, slot, 2u, rv);
  return full;
}

// Re-reads the lanes' chunks (len slots each, 0 for none), kU slots at a time, and
// buffers every nonzero that survives.  All 32 lanes call.
__device__ __forceinline__ void push_reread(const TeamArgs &A, const Team &T, Pairs &B, int &n,
                                            const RowView &rv, int32_t len, int64_t slot,
                                            int64_t elem0) {
  constexpr int kU = 4;
  const int maxlen = __reduce_max_sync(kFull, len);
  for (int k = 0; k < maxlen; k += kU) {
    double a[kU], L[kU], U[kU];
    float WU[kU], WL[kU];
    int32_t j[kU];
    uint32_t fl;
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      a[u] = 1.0;
      j[u] = 0;
      if (k + u < len) {
        a[u] = __ldg(A.M.val + elem0 + (int64_t)(k + u) * kSliceW);
        j[u] = __ldg(A.M.col + elem0 + (int64_t)(k + u) * kSliceW);
      }
    }
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      L[u] = U[u] = 0.0;
      WU[u] = WL[u] = 0.0f;
      if (k + u < len) ld_rec_l2(T.rec + j[u], L[u], U[u], WU[u], WL[u], fl);
    }
    unsigned sd[kU], some = 0u;
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      sd[u] = k + u < len ? nnz_sides(a[u], L[u], U[u], WU[u], WL[u], rv) : 0u;
      some |= sd[u];
    }
    if (__ballot_sync(kFull, some != 0u) == 0u) continue;
#pragma unroll 1
    for (int u = 0; u < kU; ++u) {
      const unsigned s = u == 0 ? sd[0] : (u == 1 ? sd[1] : (u == 2 ? sd[2] : sd[3]));
      push_pair(s != 0u, A, T, B, n, elem0 + (int64_t)(k + u) * kSliceW, slot, s, rv);
    }
  }
}

// The same for one chunk (the same in every lane) by the whole warp, a slot
// per lane.
__device__ __forceinline__ void push_reread_warp(const TeamArgs &A, const Team &T, Pairs &B,
                                                 int &n, const RowView &rv, int32_t len,
                                                 int64_t slot, int64_t elem0) {
  for (int k0 = 0; k0 < len; k0 += 32) {
    const int k = k0 + (threadIdx.x & 31);
    unsigned sides = 0u;
    if (k < len) {
      double L, U;
      float WU, WL;
      uint32_t fl;
      const double a = __ldg(A.M.val + elem0 + (int64_t)k * kSliceW);
      ld_rec_l2(T.rec + __ldg(A.M.col + elem0 + (int64_t)k * kSliceW), L, U, WU, WL, fl);
      sides = nnz_sides(a, L, U, WU, WL, rv);
    }
    push_pair(sides != 0u, A, T, B, n, elem0 + (int64_t)k * kSliceW, slot, sides, rv);
  }
}

// ----------------------------------------------------------- activities --

// A chunk before any of its nonzeros is read.
struct Head {
  int64_t c, elem0;
  int32_t len, row;  // 0 and -1 for a chunk that is not processed
  bool exact;
  double2 sd;        // {lhs, rhs}
};

__device__ __forceinline__ Head chunk_head(const TeamArgs &A, int slice, int which, bool on) {
  Head h;
  h.c = (int64_t)slice * kSliceW + which;
  const int32_t lenf = __ldg(A.M.chunk_len + h.c);
  h.row = __ldg(A.M.chunk_row + h.c);
  h.sd = __ldcg(A.side + h.c);
  h.elem0 = __ldg(A.M.slice_off + slice) + which;
  h.exact = (lenf & kExactFlag) != 0;
  h.len = lenf & kLenMask;
  if (!on || h.row < 0) {
    h.row = -1;
    h.len = 0;
    h.sd = make_double2(0.0, 0.0);
  }
  return h;
}

// Infinity counts and the screen's top-2 of a chunk.
struct Acc {
  int32_t mininf, maxinf;
  Top2 t;
};
__device__ __forceinline__ Acc acc_init() {
  Acc r;
  r.mininf = r.maxinf = 0;
  r.t = top2_init();
  return r;
}

// One nonzero's share of them; bmin, bmax: the bounds for the finite sums (0
// in the place of an infinite one).
__device__ __forceinline__ void acc_nnz(double a, double L, double U, float WU, float WL, int k,
                                        bool need_min, bool need_max, Acc &r, double &bmin,
                                        double &bmax) {
  const bool pos = d_pos(a);
  const float au = absup_fast(a), ad = absdn_fast(a);
  if (need_min) {
    const double b = pos ? L : U;
    const bool inf = d_isinf(b);
    r.mininf += inf;
    if (inf) r.t.kinf_min = k;
    bmin = inf ? 0.0 : b;
    top2_add(screen_prod(au, ad, pos ? WU : WL), k, r.t.r1, r.t.r2, r.t.kr);
  }
  if (need_max) {
    const double b = pos ? U : L;
    const bool inf = d_isinf(b);
    r.maxinf += inf;
    if (inf) r.t.kinf_max = k;
    bmax = inf ? 0.0 : b;
    top2_add(screen_prod(au, ad, pos ? WL : WU), k, r.t.l1, r.t.l2, r.t.kl);
  }
}

// Adds another part's counts and top-2.
__device__ __forceinline__ void acc_merge(Acc &r, const Acc &q) {
  if (q.mininf > 0) r.t.kinf_min = q.t.kinf_min;
  if (q.maxinf > 0) r.t.kinf_max = q.t.kinf_max;
  r.mininf += q.mininf;
  r.maxinf += q.maxinf;
  top2_merge(q.t.r1, q.t.r2, q.t.kr, r.t.r1, r.t.r2, r.t.kr);
  top2_merge(q.t.l1, q.t.l2, q.t.kl, r.t.l1, r.t.l2, r.t.kl);
}

__device__ __forceinline__ void put_partial(const TeamArgs &A, const Team &T, const Head &h,
                                            const Acc &r, double minfin, double maxfin) {
  Partial p;
  p.minfin = minfin;
  p.maxfin = maxfin;
  p.mininf = r.mininf;
  p.maxinf = r.maxinf;
  p.t = r.t;
  p.exact = h.exact ? 1 : 0;
  p.pad = 0;
  T.part[h.c] = p;
  T.touch[__ldg(A.M.chunk_sidx + h.c)] = T.round + 1;
  T.flags->touched[T.p] = 1;
}

// Step 2 and the screen thresholds of a whole row; `speaks`: one lane per row.
__device__ __forceinline__ RowView whole_row(const TeamArgs &A, const Team &T, const Head &h,
                                             const Acc &r, double minfin, double maxfin,
                                             bool speaks) {
  RowView rv;
  rv.minfin = minfin;
  rv.maxfin = maxfin;
  rv.mininf = r.mininf;
  rv.maxinf = r.maxinf;
  rv.exact = h.exact ? 1 : 0;
  rv.act = 0;
  rv.thr_r = rv.thr_l = f_inf();
  rv.lhs = h.sd.x;
  rv.rhs = h.sd.y;
  if (h.row >= 0 && row_sides_eval(rv, r.t.r1, r.t.l1, A.eps_feas) && speaks)
    T.flags->infeasible[T.p] = 1;
  return rv;
}

// One slice, a chunk per lane (those in `bits`).  This and the functions
// below that take n, the warp's buffered pairs, return the new n.
__device__ __noinline__ int slice_by_lanes(const TeamArgs &A, const Team &T, Pairs &B, int n,
                                           int slice, uint32_t bits) {
  constexpr int kG = 4;
  const int lane = threadIdx.x & 31;
  const Head h = chunk_head(A, slice, lane, ((bits >> lane) & 1u) != 0u);
  const int32_t len = h.len;
  // a warp skips the activity that none of its rows needs
  const bool need_min = __any_sync(kFull, h.row >= 0 && d_isfinite(h.sd.y));
  const bool need_max = __any_sync(kFull, h.row >= 0 && d_isfinite(h.sd.x));
  const double *vp = A.M.val + h.elem0;
  const int32_t *cp = A.M.col + h.elem0;
  double minfin = 0.0, maxfin = 0.0;
  Acc r = acc_init();
  // groups of kG slots: the gathers of a group are issued together, and the
  // next group's values and columns load behind them
  double an[kG];
  int32_t jn[kG];
#pragma unroll
  for (int u = 0; u < kG; ++u) {
    an[u] = 1.0;
    jn[u] = 0;
    if (u < len) {
      an[u] = __ldcs(vp + u * kSliceW);
      jn[u] = __ldcs(cp + u * kSliceW);
    }
  }
  for (int k = 0; k < len; k += kG) {
    double a[kG], L[kG], U[kG];
    float WU[kG], WL[kG];
    uint32_t fl[kG];
#pragma unroll
    for (int u = 0; u < kG; ++u) {
      a[u] = an[u];
      L[u] = U[u] = 0.0;
      WU[u] = WL[u] = 0.0f;
      if (k + u < len) ld_rec_l2(T.rec + jn[u], L[u], U[u], WU[u], WL[u], fl[u]);
    }
    if (k + kG < len) {
#pragma unroll
      for (int u = 0; u < kG; ++u) {
        an[u] = 1.0;
        jn[u] = 0;
        if (k + kG + u < len) {
          an[u] = __ldcs(vp + (int64_t)(k + kG + u) * kSliceW);
          jn[u] = __ldcs(cp + (int64_t)(k + kG + u) * kSliceW);
        }
      }
    }
#pragma unroll
    for (int u = 0; u < kG; ++u) {
      if (k + u < len) {
        double bmin, bmax;
        acc_nnz(a[u], L[u], U[u], WU[u], WL[u], k + u, need_min, false, r, bmin, bmax);
        if (need_min) minfin = fma(a[u], bmin, minfin);
        acc_nnz(a[u], L[u], U[u], WU[u], WL[u], k + u, false, need_max, r, bmin, bmax);
        if (need_max) maxfin = fma(a[u], bmax, maxfin);
      }
    }
  }
  if (h.exact) r.t.r1 = r.t.r2 = r.t.l1 = r.t.l2 = f_inf();
  if (slice < A.M.nslices_split) {  // warp-uniform
    if (h.row >= 0) put_partial(A, T, h, r, minfin, maxfin);
    return n;
  }
  const RowView rv = whole_row(A, T, h, r, minfin, maxfin, true);
  const bool full = push_named(A, T, B, n, rv, r.t, r.mininf, r.maxinf, h.c, h.elem0);
  if (__ballot_sync(kFull, full) != 0u)
    push_reread(A, T, B, n, rv, full ? len : 0, h.c, h.elem0);
  return n;
}

// A slice of rows of at most kMax nonzeros: the survivors come from the
// screen values the lanes keep, without a second pass.
template <int kSides, int kMax>
__device__ __forceinline__ int short_rows(const TeamArgs &A, const Team &T, Pairs &B, int n,
                                          const Head &h, bool right) {
  ShortAct<kSides, kMax> r;
  short_activity<kSides, kMax>(
      A.M, h.elem0, h.len, right,
      [&](int32_t j, double &L, double &U, float &WU, float &WL) {
        uint32_t fl;
        ld_rec_l2(T.rec + j, L, U, WU, WL, fl);
      },
      r);
  constexpr int kR = 0, kL = kSides - 1;  // one side: both names are its index
  const bool use_r = kSides == 2 || right, use_l = kSides == 2 || !right;
  Acc q = acc_init();
  q.mininf = use_r ? r.ninf[kR] : 0;
  q.maxinf = use_l ? r.ninf[kL] : 0;
  if (use_r) q.t.r1 = h.exact ? f_inf() : short_max(r.t[kR]);
  if (use_l) q.t.l1 = h.exact ? f_inf() : short_max(r.t[kL]);
  const RowView rv = whole_row(A, T, h, q, use_r ? r.fin[kR] : 0.0, use_l ? r.fin[kL] : 0.0, true);
  uint32_t mr = 0u, ml = 0u;
  if (rv.act) {
    if (use_r)
      mr = short_survivors(r.t[kR], h.len, d_isfinite(rv.rhs), rv.mininf, r.kinf[kR], rv.thr_r,
                           h.exact);
    if (use_l)
      ml = short_survivors(r.t[kL], h.len, d_isfinite(rv.lhs), rv.maxinf, r.kinf[kL], rv.thr_l,
                           h.exact);
  }
  for (uint32_t m = mr | ml; __any_sync(kFull, m != 0u); m &= m - 1u) {
    const int k = m != 0u ? __ffs(m) - 1 : 0;
    push_pair(m != 0u, A, T, B, n, h.elem0 + k * kSliceW, h.c,
              ((mr >> k) & 1u) | (((ml >> k) & 1u) << 1), rv);
  }
  return n;
}

template <int kMax>
__device__ __noinline__ int slice_short(const TeamArgs &A, const Team &T, Pairs &B, int n,
                                        int slice, uint32_t bits) {
  const int lane = threadIdx.x & 31;
  const Head h = chunk_head(A, slice, lane, ((bits >> lane) & 1u) != 0u);
  const bool need_min = __any_sync(kFull, h.row >= 0 && d_isfinite(h.sd.y));
  const bool need_max = __any_sync(kFull, h.row >= 0 && d_isfinite(h.sd.x));
  if (need_min && need_max) return short_rows<2, kMax>(A, T, B, n, h, true);
  return short_rows<1, kMax>(A, T, B, n, h, need_min);
}

// One chunk by the whole warp: the lanes gather 32 slots side by side, and
// the chain runs over shuffled values (the lanes below 16 add up the minimum
// activity, the others the maximum): the same FMA chain in CSR order at 64
// clocks per slot, where a lane alone takes about 310.
__device__ __noinline__ int chunk_by_warp(const TeamArgs &A, const Team &T, Pairs &B, int n,
                                          int slice, int which) {
  const int lane = threadIdx.x & 31;
  const Head h = chunk_head(A, slice, which, true);
  if (h.row < 0) return n;  // warp-uniform
  const bool need_min = d_isfinite(h.sd.y), need_max = d_isfinite(h.sd.x);
  double fin = 0.0;
  Acc r = acc_init();
  for (int t0 = 0; t0 < h.len; t0 += 128) {
    double a[4], bmin[4], bmax[4], L[4], U[4];
    float WU[4], WL[4];
    int32_t j[4];
    uint32_t fl;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int k = t0 + 32 * u + lane;
      a[u] = 1.0;
      j[u] = 0;
      bmin[u] = bmax[u] = 0.0;
      if (k < h.len) {
        a[u] = __ldg(A.M.val + h.elem0 + (int64_t)k * kSliceW);
        j[u] = __ldg(A.M.col + h.elem0 + (int64_t)k * kSliceW);
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (t0 + 32 * u + lane < h.len) ld_rec_l2(T.rec + j[u], L[u], U[u], WU[u], WL[u], fl);
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (t0 + 32 * u + lane < h.len)
        acc_nnz(a[u], L[u], U[u], WU[u], WL[u], t0 + 32 * u + lane, need_min, need_max, r,
                bmin[u], bmax[u]);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int m = min(32, h.len - t0 - 32 * u);
#pragma unroll 4
      for (int i = 0; i < m; ++i) {  // warp-uniform
        const double av = __shfl_sync(kFull, a[u], i);
        const double bn = __shfl_sync(kFull, bmin[u], i), bx = __shfl_sync(kFull, bmax[u], i);
        fin = fma(av, lane < 16 ? bn : bx, fin);
      }
    }
  }
  const double minfin = need_min ? __shfl_sync(kFull, fin, 0) : 0.0;
  const double maxfin = need_max ? __shfl_sync(kFull, fin, 16) : 0.0;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    Acc q;
    q.mininf = __shfl_xor_sync(kFull, r.mininf, o);
    q.maxinf = __shfl_xor_sync(kFull, r.maxinf, o);
    q.t.kinf_min = __shfl_xor_sync(kFull, r.t.kinf_min, o);
    q.t.kinf_max = __shfl_xor_sync(kFull, r.t.kinf_max, o);
    q.t.r1 = __shfl_xor_sync(kFull, r.t.r1, o);
    q.t.r2 = __shfl_xor_sync(kFull, r.t.r2, o);
    q.t.l1 = __shfl_xor_sync(kFull, r.t.l1, o);
    q.t.l2 = __shfl_xor_sync(kFull, r.t.l2, o);
    q.t.kr = __shfl_xor_sync(kFull, r.t.kr, o);
    q.t.kl = __shfl_xor_sync(kFull, r.t.kl, o);
    acc_merge(r, q);
  }
  if (h.exact) r.t.r1 = r.t.r2 = r.t.l1 = r.t.l2 = f_inf();
  if (slice < A.M.nslices_split) {
    if (lane == 0) put_partial(A, T, h, r, minfin, maxfin);
    return n;
  }
  RowView rv = whole_row(A, T, h, r, minfin, maxfin, lane == 0);
  if (rv.act == 0) return n;  // warp-uniform
  if (lane != 0) rv.act = 0;  // one lane speaks for the row
  const bool full = __shfl_sync(
      kFull, push_named(A, T, B, n, rv, r.t, r.mininf, r.maxinf, h.c, h.elem0), 0);
  if (!full) return n;
  push_reread_warp(A, T, B, n, rv, h.len, h.c, h.elem0);
  return n;
}

// Marked chunks up to which a long slice is processed chunk by chunk.
constexpr int kByWarp = 2;
// Longest row whose screen values stay in registers here (128 a thread).
constexpr int kMidRow = 24;
// Chunks of long slices (kLongSlots slots and more) per warp up to which they
// all are: a lane's walk of 256 slots takes 45 us, a warp's 12 us.
constexpr int kChunksPerWarp = 4;

__device__ __forceinline__ int do_slice(const TeamArgs &A, const Team &T, Pairs &B, int n,
                                        int slice, uint32_t bits) {
  const int32_t len = __ldg(A.M.slice_len + slice);
  if (len <= kMidRow && slice >= A.M.nslices_split)
    return len <= kShortRow ? slice_short<kShortRow>(A, T, B, n, slice, bits)
                            : slice_short<kMidRow>(A, T, B, n, slice, bits);
  if (__popc(bits) > kByWarp || len < 16) return slice_by_lanes(A, T, B, n, slice, bits);
  for (; bits != 0u; bits &= bits - 1u) n = chunk_by_warp(A, T, B, n, slice, __ffs(bits) - 1);
  return n;
}

// ---------------------------------------------------------- split rows --

struct RowAcc {
  double mnf, mxf;
  int32_t mni, mxi, ex;
  float Tr, Tl;
};
__device__ __forceinline__ RowAcc rowacc_init() {
  RowAcc a;
  a.mnf = a.mxf = 0.0;
  a.mni = a.mxi = a.ex = 0;
  a.Tr = a.Tl = -f_inf();
  return a;
}
__device__ __forceinline__ void rowacc_add(RowAcc &a, const Partial &p) {
  a.mnf += p.minfin;
  a.mxf += p.maxfin;
  a.mni += p.mininf;
  a.mxi += p.maxinf;
  a.Tr = fmaxf(a.Tr, p.t.r1);
  a.Tl = fmaxf(a.Tl, p.t.l1);
  a.ex |= p.exact;
}
__device__ __forceinline__ Partial ld_partial(const Partial *p) {
  union {
    Partial x;
    int4 w[sizeof(Partial) / 16];
  } u;
#pragma unroll
  for (int k = 0; k < (int)(sizeof(Partial) / 16); ++k)
    u.w[k] = __ldcg(reinterpret_cast<const int4 *>(p) + k);
  return u.x;
}

// Pieces q, q + step, ... below e in that order, four loads in flight.
__device__ __forceinline__ void rowacc_run(const TeamArgs &A, const Team &T, int32_t q, int32_t e,
                                           int32_t step, RowAcc &a) {
  for (; q < e; q += 4 * step) {
    Partial p[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (q + u * step < e) p[u] = ld_partial(T.part + __ldg(A.M.split_cidx + q + u * step));
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (q + u * step < e) rowacc_add(a, p[u]);
  }
}

constexpr int kCombineShort = 4;  // as the graph's k_combine
constexpr int kCombineSpans = 8;  // as the batched nodes' k_bcombine

// Step 2 and the thresholds of split row w from its sums (one lane).
__device__ __forceinline__ void split_commit(const TeamArgs &A, const Team &T, int32_t w,
                                             int32_t first, RowAcc &a) {
  const double2 sd = __ldcg(A.side + __ldg(A.M.split_cidx + first));
  RowView rv;
  rv.minfin = a.mnf;
  rv.maxfin = a.mxf;
  rv.mininf = a.mni;
  rv.maxinf = a.mxi;
  rv.lhs = sd.x;
  rv.rhs = sd.y;
  rv.exact = a.ex;
  if (a.ex) a.Tr = a.Tl = f_inf();
  if (row_sides_eval(rv, a.Tr, a.Tl, A.eps_feas)) T.flags->infeasible[T.p] = 1;
  RowTot rt;
  rt.minfin = a.mnf;
  rt.maxfin = a.mxf;
  rt.mininf = a.mni;
  rt.maxinf = a.mxi;
  rt.thr_r = rv.thr_r;
  rt.thr_l = rv.thr_l;
  rt.active = rv.act ? T.round + 1 : 0;
  rt.row = 0;
  T.rowtot[w] = rt;
}

// Sums of the split rows that had a piece recomputed this round.  The
// association is that of the other kernels for the same kind of call: rows
// of few pieces in piece order; else, for single problems and sets, lanes
// strided over the pieces and a butterfly, and for nodes contiguous eighths
// added in order.
__device__ __noinline__ void combine_rows(const TeamArgs &A, const Team &T) {
  const int lane = threadIdx.x & 31;
  const int now = T.round + 1;
  const int32_t r0 = T.v.srow0, r1 = T.v.srow1;
  for (int32_t r = r0 + T.gw() * 32 + lane; r < r1; r += T.nw * 32) {  // short rows by lane
    const int32_t cb = __ldg(A.M.split_cbeg + r), ce = __ldg(A.M.split_cbeg + r + 1);
    if (ce - cb > kCombineShort || __ldcg(T.touch + r) != now) continue;
    RowAcc a = rowacc_init();
    rowacc_run(A, T, cb, ce, 1, a);
    split_commit(A, T, r, cb, a);
  }
  for (int32_t r = r0 + T.gw(); r < r1; r += T.nw) {  // long rows by warp
    const int32_t cb = __ldg(A.M.split_cbeg + r), ce = __ldg(A.M.split_cbeg + r + 1);
    if (ce - cb <= kCombineShort || __ldcg(T.touch + r) != now) continue;
    RowAcc a = rowacc_init();
    if (A.node_sums) {
      const int32_t span = (ce - cb + kCombineSpans - 1) / kCombineSpans;
      const int32_t qa = min(ce, cb + lane * span);
      if (lane < kCombineSpans) rowacc_run(A, T, qa, min(ce, qa + span), 1, a);
      RowAcc t = rowacc_init();
#pragma unroll
      for (int k = 0; k < kCombineSpans; ++k) {
        t.mnf += __shfl_sync(kFull, a.mnf, k);
        t.mxf += __shfl_sync(kFull, a.mxf, k);
        t.mni += __shfl_sync(kFull, a.mni, k);
        t.mxi += __shfl_sync(kFull, a.mxi, k);
        t.Tr = fmaxf(t.Tr, __shfl_sync(kFull, a.Tr, k));
        t.Tl = fmaxf(t.Tl, __shfl_sync(kFull, a.Tl, k));
        t.ex |= __shfl_sync(kFull, a.ex, k);
      }
      a = t;
    } else {
      rowacc_run(A, T, cb + lane, ce, 32, a);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        a.mnf += __shfl_xor_sync(kFull, a.mnf, o);
        a.mxf += __shfl_xor_sync(kFull, a.mxf, o);
        a.mni += __shfl_xor_sync(kFull, a.mni, o);
        a.mxi += __shfl_xor_sync(kFull, a.mxi, o);
        a.Tr = fmaxf(a.Tr, __shfl_xor_sync(kFull, a.Tr, o));
        a.Tl = fmaxf(a.Tl, __shfl_xor_sync(kFull, a.Tl, o));
        a.ex |= __shfl_xor_sync(kFull, a.ex, o);
      }
    }
    if (lane == 0) split_commit(A, T, r, cb, a);
  }
}

// Candidates of a split row's chunk by the whole warp.
__device__ __forceinline__ int split_chunk(const TeamArgs &A, const Team &T, Pairs &B, int n,
                                           int64_t c) {
  const int lane = threadIdx.x & 31;
  const int32_t s = __ldg(A.M.chunk_sidx + c);
  if (s < 0 || __ldcg(&T.rowtot[s].active) != T.round + 1) return n;  // warp-uniform
  const RowTot *q = T.rowtot + s;
  const Partial p = ld_partial(T.part + c);
  const double2 f = __ldcg(reinterpret_cast<const double2 *>(&q->minfin));
  const int4 w = __ldcg(reinterpret_cast<const int4 *>(&q->mininf));
  const double2 sd = __ldcg(A.side + c);
  const int32_t lenf = __ldg(A.M.chunk_len + c), len = lenf & kLenMask;
  RowView rv;
  rv.minfin = f.x;
  rv.maxfin = f.y;
  rv.mininf = w.x;
  rv.maxinf = w.y;
  rv.thr_r = __int_as_float(w.z);
  rv.thr_l = __int_as_float(w.w);
  rv.lhs = sd.x;
  rv.rhs = sd.y;
  rv.exact = (lenf & kExactFlag) ? 1 : 0;
  rv.act = lane == 0 ? 1 : 0;  // one lane speaks for the chunk
  const int64_t elem0 = __ldg(A.M.slice_off + c / kSliceW) + c % kSliceW;
  if (__shfl_sync(kFull, push_named(A, T, B, n, rv, p.t, p.mininf, p.maxinf, c, elem0), 0))
    push_reread_warp(A, T, B, n, rv, len, c, elem0);
  return n;
}

// Candidates of the split rows that may have one: every chunk of such a row.
__device__ __noinline__ int split_candidates(const TeamArgs &A, const Team &T, Pairs &B,
                                             int n, bool by_chunk) {
  const int lane = threadIdx.x & 31;
  int first = T.v.split0;
  if (by_chunk) {
    first += T.v.nlsplit;
    for (int x = T.gw(); x < T.v.nlsplit * kSliceW; x += T.nw)
      n = split_chunk(A, T, B, n, (int64_t)T.v.split0 * kSliceW + x);
  }
  for (int slice = first + T.gw(); slice < T.v.split1; slice += T.nw) {
    const int64_t c = (int64_t)slice * kSliceW + lane;
    const int32_t s = __ldg(A.M.chunk_sidx + c);
    const bool on = s >= 0 && __ldcg(&T.rowtot[s].active) == T.round + 1;
    if (__ballot_sync(kFull, on) == 0u) continue;
    RowView rv;
    rv.act = rv.exact = rv.mininf = rv.maxinf = 0;
    rv.minfin = rv.maxfin = rv.lhs = rv.rhs = 0.0;
    rv.thr_r = rv.thr_l = f_inf();
    Top2 t = top2_init();
    int32_t len = 0, cmin = 0, cmax = 0;
    if (on) {
      const RowTot *q = T.rowtot + s;
      const Partial p = ld_partial(T.part + c);
      const double2 f = __ldcg(reinterpret_cast<const double2 *>(&q->minfin));
      const int4 w = __ldcg(reinterpret_cast<const int4 *>(&q->mininf));
      const double2 sd = __ldcg(A.side + c);
      const int32_t lenf = __ldg(A.M.chunk_len + c);
      len = lenf & kLenMask;
      rv.minfin = f.x;
      rv.maxfin = f.y;
      rv.mininf = w.x;
      rv.maxinf = w.y;
      rv.thr_r = __int_as_float(w.z);
      rv.thr_l = __int_as_float(w.w);
      rv.lhs = sd.x;
      rv.rhs = sd.y;
      rv.exact = (lenf & kExactFlag) ? 1 : 0;
      rv.act = 1;
      t = p.t;
      cmin = p.mininf;
      cmax = p.maxinf;
    }
    const int64_t elem0 = __ldg(A.M.slice_off + slice) + lane;
    const bool full = push_named(A, T, B, n, rv, t, cmin, cmax, c, elem0);
    if (__ballot_sync(kFull, full) == 0u) continue;
    push_reread(A, T, B, n, rv, full ? len : 0, c, elem0);
  }
  return n;
}

// --------------------------------------------------------------- commit --

// A round that changes more than a kMarkShare-th of the variables is followed
// by one that processes every chunk: marking costs an atomic per nonzero of
// the changed variables, and at that share most rows are marked anyway.
constexpr int kMarkShare = 12;
constexpr int32_t kMarkAlways = 1 << 15;  // fewer variables: always marked
constexpr int kCommitWords = 8;           // most dirty words per warp and step

// Ends a round: the changed variables' keys become their records, crossing
// bounds are infeasible, and the variables' chunks are marked for the next
// round.  A warp takes kCommitWords words of the dirty bitmap and then their
// variables 32 at a time.
__device__ __noinline__ void commit_round(const TeamArgs &A, const Team &T, float tau_dn,
                                             float eps_dn) {
  const int lane = threadIdx.x & 31;
  const int32_t nv = T.v.var1 - T.v.var0;
  const int64_t words = ((int64_t)nv + 31) >> 5;
  // this round's masks are read: the next round marks in them
  const int ns = T.v.split1 - T.v.split0, nsl = ns + (T.v.whole1 - T.v.whole0);
  for (int q = T.gw() * 32 + lane; q < nsl; q += T.nw * 32)
    T.mask[T.p * T.nmask + (q < ns ? T.v.split0 + q : T.v.whole0 + (q - ns))] = 0u;
  const int32_t limit = nv <= kMarkAlways ? nv : nv / kMarkShare;
  // as few words per warp as give every warp some
  const int64_t share = words / T.nw;
  const int per = share < 1 ? 1 : (share > kCommitWords ? kCommitWords : (int)share);
  for (int64_t w0 = (int64_t)T.gw() * per; w0 < words; w0 += (int64_t)T.nw * per) {
    uint32_t bits = 0u;
    if (lane < per && w0 + lane < words) {
      uint32_t *q = T.dirty + T.v.dword0 + w0 + lane;
      bits = __ldcg(q);
      if (bits) *q = 0u;
    }
    if (__ballot_sync(kFull, bits != 0u) == 0u) continue;
    int incl = __popc(bits);  // of the first kCommitWords lanes
#pragma unroll
    for (int o = 1; o < kCommitWords; o <<= 1) {
      const int v = __shfl_up_sync(kFull, incl, o);
      if (lane >= o) incl += v;
    }
    const int total = __shfl_sync(kFull, incl, kCommitWords - 1);
    bool mark = true;
    if (nv > kMarkAlways) {
      int32_t before = 0;
      if (lane == 0) before = atomicAdd(&T.flags->nchanged[T.p], total);
      mark = __shfl_sync(kFull, before, 0) <= limit;
      if (!mark && lane == 0) T.flags->all_next[T.p] = 1;
    }
    for (int b0 = 0; b0 < total; b0 += 32) {
      const int k = b0 + lane;
      int src = 0;  // the word that holds the k-th changed variable
#pragma unroll
      for (int o = kCommitWords / 2; o > 0; o >>= 1) {
        const int v = __shfl_sync(kFull, incl, src + o - 1);
        if (v <= k) src += o;
      }
      src &= kCommitWords - 1;
      const uint32_t wd = __shfl_sync(kFull, bits, src);
      const int below = __shfl_sync(kFull, incl, src) - __popc(wd);
      int32_t beg = 0, deg = 0;
      if (k < total) {
        const int64_t j = T.v.var0 + (w0 + src) * 32 + nth_bit(wd, k - below);
        const longlong2 kk = __ldcg(T.keys + j);
        const bool isint = __ldg(A.vt + j) != 0;
        if (mark) {
          beg = __ldg(A.M.col_ptr + j);
          deg = __ldg(A.M.col_ptr + j + 1) - beg;
        }
        const double L = val_of_key(kk.x), U = val_of_key(kk.y);
        if (kk.x > kk.y) {  // L > U in key order: test the crossing exactly
          const bool cross = isint ? (L > U) : (L > U + A.eps_feas * d_max1abs(U));
          if (cross) T.flags->infeasible[T.p] = 1;
        }
        put_var(T.rec + j, L, U, isint, tau_dn, eps_dn);
      }
      if (!markable(deg)) {
        if (lane == 0) T.flags->all_next[T.p] = 1;
      } else if (mark) {
        mark_columns<true>(A.M.col_slot, T.mask + (T.p ^ 1) * T.nmask, beg, deg);
      }
    }
  }
}

// ------------------------------------------------------------- prologue --

// Normalises one item's inputs into the team's state: |v| >= inf_thr becomes
// +-inf, integer bounds are rounded; NaN and contradictory infinities set
// the error word.
__device__ __noinline__ void begin_item(const TeamArgs &A, const Team &T, int item,
                                           float tau_dn, float eps_dn) {
  const double pinf = __longlong_as_double(0x7FF0000000000000ll), thr = A.inf_thr;
  const long long k_thr = cmp_key(thr), k_mthr = cmp_key(-thr);
  const int lane = threadIdx.x & 31;
  const int32_t nv = T.v.var1 - T.v.var0;
  const double *lb = A.lb + (int64_t)item * A.in_stride, *ub = A.ub + (int64_t)item * A.in_stride;
  bool bad = false;
  for (int64_t i0 = (int64_t)T.gw() * 32; i0 < nv; i0 += (int64_t)T.nw * 32) {
    const int64_t i = i0 + lane, j = T.v.var0 + i;
    bool cross = false;
    if (i < nv) {
      double L = lb[j], U = ub[j];
      const bool isint = A.vt[j] != 0;
      if (d_isnan(L) || d_isnan(U) || cmp_key(L) >= k_thr || cmp_key(U) <= k_mthr) {
        bad = true;
        L = U = 0.0;
      }
      if (cmp_key(L) <= k_mthr) L = -pinf;
      if (cmp_key(U) >= k_thr) U = pinf;
      if (isint) {
        if (d_isfinite(L)) L = d_ceil_int(L - A.eps_int);
        if (d_isfinite(U)) U = d_floor_int(U + A.eps_int);
      }
      T.keys[j] = make_longlong2(key_of(L), key_of(U));
      put_var(T.rec + j, L, U, isint, tau_dn, eps_dn);
      cross = key_of(L) > key_of(U);
    }
    // bounds that cross on input are committed, and so tested, in round 1
    const unsigned cw = __ballot_sync(kFull, cross);
    if (lane == 0) T.dirty[T.v.dword0 + (i0 >> 5)] = cw;
  }
  const int ns = T.v.split1 - T.v.split0, nsl = ns + (T.v.whole1 - T.v.whole0);
  for (int q = T.gw(); q < nsl; q += T.nw) {
    const int slice = q < ns ? T.v.split0 + q : T.v.whole0 + (q - ns);
    if (lane < 2) T.mask[lane * T.nmask + slice] = 0u;
    if (!A.sides_ready) {
      const int64_t c = (int64_t)slice * kSliceW + lane;
      const int32_t row = __ldg(A.M.chunk_row + c);
      double l = 0.0, r = 0.0;
      if (row >= 0) {
        l = A.lhs[row];
        r = A.rhs[row];
        if (d_isnan(l) || d_isnan(r) || cmp_key(l) >= k_thr || cmp_key(r) <= k_mthr) {
          bad = true;
          l = r = 0.0;
        }
        if (cmp_key(l) <= k_mthr) l = -pinf;
        if (cmp_key(r) >= k_thr) r = pinf;
      }
      A.side[c] = make_double2(l, r);
    }
  }
  for (int32_t r = T.v.srow0 + T.gw() * 32 + lane; r < T.v.srow1; r += T.nw * 32) {
    T.touch[r] = 0;
    T.rowtot[r].active = 0;
  }
  if (bad) atomicExch(&T.flags->err, DP_ERR_NAN_INPUT);
}

// --------------------------------------------------------------- kernel --

__global__ void __launch_bounds__(kThreads, 2) k_team(const __grid_constant__ TeamArgs A) {
  __shared__ Pairs s_pairs[kWarps];
  __shared__ Team T;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  Pairs &B = s_pairs[warp];
  unsigned cr, cn;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(cr));
  asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(cn));
  const int rank = (int)cr, nb = (int)cn;
  const int team = blockIdx.x / nb, teams = gridDim.x / nb;
  const int gw = warp * nb + rank;
  if (threadIdx.x == 0) {
    T.rank = rank;
    T.nb = nb;
    T.nw = nb * kWarps;
    T.rec = A.rec + team * A.s_var;
    T.keys = A.keys + team * A.s_var;
    T.dirty = A.dirty + team * A.s_dirty;
    T.mask = A.mask + team * A.s_mask;
    T.nmask = A.M.nslices;
    T.touch = A.touch + team * A.s_touch;
    T.part = A.part + team * A.s_part;
    T.rowtot = A.rowtot + team * A.s_touch;
    T.flags = A.flags + team;
  }
  const float tau_dn = f32_dn(A.tau_rel), eps_dn = f32_dn(A.eps_int);
  const bool leader = rank == 0 && threadIdx.x == 0;

  for (int item = team; item < A.count;) {
    if (threadIdx.x == 0) {
      if (A.views) {
        T.v = A.views[item];
      } else {
        T.v.split0 = 0;
        T.v.split1 = T.v.whole0 = A.M.nslices_split;
        T.v.whole1 = A.M.nslices;
        T.v.srow0 = 0;
        T.v.srow1 = A.M.nsplit_rows;
        T.v.var0 = 0;
        T.v.var1 = A.M.n;
        T.v.dword0 = 0;
        T.v.nlsplit = A.M.long_split;
        T.v.nlwhole = A.M.long_whole;
        T.v.id = item;
      }
      T.round = 0;
      T.p = 0;
    }
    __syncthreads();
    int round = 0;
    if (leader) {
#pragma unroll
      for (int k = 0; k < 2; ++k)
        T.flags->changed[k] = T.flags->infeasible[k] = T.flags->touched[k] =
            T.flags->all_next[k] = T.flags->nchanged[k] = 0;
      if (teams < A.count) T.flags->item = teams + atomicAdd(A.next, 1);
    }
    begin_item(A, T, item, tau_dn, eps_dn);
    cluster_barrier();
    const int32_t err = __ldcg(&T.flags->err);
    int32_t infeasible = 0, changed = 0;
    bool all = true;
    const int ns = T.v.split1 - T.v.split0, nsl = ns + (T.v.whole1 - T.v.whole0);
    const int nl = T.v.nlsplit + T.v.nlwhole;
    const bool by_chunk = nl * kSliceW <= kChunksPerWarp * T.nw;
    if (err == 0 && A.max_rounds > 0) {
      for (;;) {
        const int p = round & 1;
        int n = 0;
        const uint32_t *mask = T.mask + p * T.nmask;
        // items: the chunks of the long slices (a warp each), then the other
        // slices; a warp looks at 32 of its items at a time, its turn reversed
        // in every other pass (slices are sorted by length)
        const int skip = by_chunk ? nl : 0, skip_split = by_chunk ? T.v.nlsplit : 0;
        const int chunks = skip * kSliceW, items = chunks + nsl - skip;
        for (int q0 = 0; q0 * T.nw < items; q0 += 32) {
          const int pass = q0 + lane;
          const int64_t q = (int64_t)pass * T.nw + ((pass & 1) ? T.nw - 1 - gw : gw);
          int slice = 0;
          uint32_t bits = 0u;
          if (q < chunks) {
            const int x = (int)q / kSliceW;
            slice = x < skip_split ? T.v.split0 + x : T.v.whole0 + (x - skip_split);
            bits = (all ? kFull : __ldcg(mask + slice)) & (1u << (q % kSliceW));
          } else if (q < items) {
            const int x = (int)q - chunks + skip_split;  // the split slices that remain first
            slice = x < ns ? T.v.split0 + x : T.v.whole0 + (skip - skip_split) + (x - ns);
            bits = all ? kFull : __ldcg(mask + slice);
          }
          unsigned todo = __ballot_sync(kFull, bits != 0u);
          for (; todo != 0u; todo &= todo - 1u) {
            const int src = __ffs(todo) - 1;
            n = do_slice(A, T, B, n, __shfl_sync(kFull, slice, src), __shfl_sync(kFull, bits, src));
          }
        }
        if (T.v.srow1 > T.v.srow0) {
          cluster_barrier();
          if (__ldcg(&T.flags->touched[p])) {
            combine_rows(A, T);
            cluster_barrier();
            n = split_candidates(A, T, B, n, by_chunk);
          }
        }
        if (n > 0) eval_pairs(A, T, B, 0, n);
        cluster_barrier();
        if (leader) {  // the next round's words, last read before this round began
          T.flags->changed[p ^ 1] = 0;
          T.flags->infeasible[p ^ 1] = 0;
          T.flags->touched[p ^ 1] = 0;
          T.flags->all_next[p ^ 1] = 0;
          T.flags->nchanged[p ^ 1] = 0;
        }
        commit_round(A, T, tau_dn, eps_dn);
        cluster_barrier();
        changed = __ldcg(&T.flags->changed[p]);
        infeasible = __ldcg(&T.flags->infeasible[p]);
        all = __ldcg(&T.flags->all_next[p]) != 0;
        ++round;
        if (!changed || infeasible || round >= A.max_rounds) break;
        if (threadIdx.x == 0) {  // no thread of the block is past the barrier below
          T.round = round;
          T.p = round & 1;
        }
        __syncthreads();
      }
    }
    // outputs (an item with bad inputs has none)
    if (err == 0) {
      double *lo = A.lb_out + (int64_t)item * A.in_stride;
      double *hi = A.ub_out + (int64_t)item * A.in_stride;
      for (int64_t j = T.v.var0 + (int64_t)gw * 32 + lane; j < T.v.var1; j += (int64_t)T.nw * 32) {
        const longlong2 kk = __ldcg(T.keys + j);
        lo[j] = val_of_key(kk.x);
        hi[j] = val_of_key(kk.y);
      }
    }
    if (leader)
      A.res[T.v.id] = make_int4(infeasible, round,
                              (!infeasible && changed && round >= A.max_rounds) ? 1 : 0, err);
    int next = item + teams;
    if (teams < A.count) next = __ldcg(&T.flags->item);
    else next = A.count;
    // the state is free for the next item once every block is done with it
    if (next < A.count || err != 0)
      cluster_barrier();
    if (err != 0 && leader) T.flags->err = 0;
    if (next < A.count && err != 0)
      cluster_barrier();
    item = next;
  }
}

// Sides in slot order for a call whose teams share them.
__global__ void __launch_bounds__(kThreads)
k_team_sides(const __grid_constant__ TeamArgs A) {
  const double pinf = __longlong_as_double(0x7FF0000000000000ll), thr = A.inf_thr;
  const int64_t nslots = (int64_t)A.M.nslices * kSliceW;
  for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < nslots;
       c += (int64_t)gridDim.x * blockDim.x) {
    const int32_t row = A.M.chunk_row[c];
    double l = 0.0, r = 0.0;
    if (row >= 0) {
      l = A.lhs[row];
      r = A.rhs[row];
      // any team reports it
      if (d_isnan(l) || d_isnan(r) || l >= thr || r <= -thr) {
        atomicExch(&A.flags->err, DP_ERR_NAN_INPUT);
        l = r = 0.0;
      }
      if (l <= -thr) l = -pinf;
      if (r >= thr) r = pinf;
    }
    A.side[c] = make_double2(l, r);
  }
}

// -------------------------------------------------------- column lists --
//
// Built on the device when a matrix is loaded: nonzeros counted per column,
// the counts summed up, and every nonzero's chunk slot stored at its column's
// cursor (the order within a column does not matter: marking ORs bits).

template <bool kFill>
__global__ void __launch_bounds__(kThreads)
k_columns(DevMatrix M, int32_t *count, int32_t *col_slot) {
  const int lane = threadIdx.x & 31;
  const int nw = gridDim.x * kWarps;
  for (int slice = blockIdx.x * kWarps + (threadIdx.x >> 5); slice < M.nslices; slice += nw) {
    const int32_t slot = slice * kSliceW + lane;
    const int32_t len = M.chunk_len[slot] & kLenMask;
    const int32_t *cp = M.col + M.slice_off[slice] + lane;
    for (int32_t k = 0; k < len; ++k) {
      const int32_t at = atomicAdd(&count[cp[(int64_t)k * kSliceW]], 1);
      if (kFill) col_slot[at] = slot;
    }
  }
}

// Exclusive sums of count[0, n) in place and into ptr[0, n]; one block.
__global__ void __launch_bounds__(1024) k_column_sums(int32_t n, int32_t *count, int32_t *ptr) {
  __shared__ int32_t s_warp[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int32_t run = 0;
  for (int64_t j0 = 0; j0 < n; j0 += 1024) {
    const int64_t j = j0 + threadIdx.x;
    const int32_t v = j < n ? count[j] : 0;
    int32_t incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t u = __shfl_up_sync(kFull, incl, o);
      if (lane >= o) incl += u;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    int32_t base = 0, all = 0;
    for (int q = 0; q < 32; ++q) {
      if (q < warp) base += s_warp[q];
      all += s_warp[q];
    }
    if (j < n) {
      count[j] = run + base + incl - v;
      ptr[j] = run + base + incl - v;
    }
    run += all;
    __syncthreads();
  }
  if (threadIdx.x == 0) ptr[n] = run;
}

}  // namespace

cudaError_t launch_columns(const DevMatrix &M, int32_t *count, int32_t *col_ptr,
                           int32_t *col_slot, int num_sms, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(count, 0, sizeof(int32_t) * (size_t)(M.n > 0 ? M.n : 1), st);
  if (e != cudaSuccess) return e;
  const int nb = num_sms * 8;
  k_columns<false><<<nb, kThreads, 0, st>>>(M, count, nullptr);
  k_column_sums<<<1, 1024, 0, st>>>(M.n, count, col_ptr);
  k_columns<true><<<nb, kThreads, 0, st>>>(M, count, col_slot);
  return cudaGetLastError();
}

namespace {
cudaLaunchConfig_t cluster_config(int blocks, int size, cudaStream_t st,
                                  cudaLaunchAttribute *attr) {
  cudaLaunchConfig_t c = {};
  c.gridDim = dim3(blocks);
  c.blockDim = dim3(kThreads);
  c.stream = st;
  attr->id = cudaLaunchAttributeClusterDimension;
  attr->val.clusterDim.x = size;
  attr->val.clusterDim.y = attr->val.clusterDim.z = 1;
  c.attrs = attr;
  c.numAttrs = 1;
  return c;
}
}  // namespace

int cluster_teams_resident(int size) {
  if (size > 8 && cudaFuncSetAttribute(k_team, cudaFuncAttributeNonPortableClusterSizeAllowed,
                                       1) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  cudaLaunchAttribute attr[1];
  const cudaLaunchConfig_t c = cluster_config(size, size, nullptr, attr);
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, k_team, &c) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}

cudaError_t launch_cluster_teams(const TeamArgs &A, int teams, int size, int num_sms,
                                 cudaStream_t st) {
  cudaError_t e;
  if (A.sides_ready) {  // shared by the teams: written first
    const int64_t want = ((int64_t)A.M.nslices * kSliceW + kThreads - 1) / kThreads;
    const int nb = (int)(want < 1 ? 1 : (want > num_sms * 8 ? num_sms * 8 : want));
    k_team_sides<<<nb, kThreads, 0, st>>>(A);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  if (teams < A.count &&
      (e = cudaMemsetAsync(A.next, 0, sizeof(int32_t), st)) != cudaSuccess)
    return e;
  cudaLaunchAttribute attr[1];
  const cudaLaunchConfig_t c = cluster_config(teams * size, size, st, attr);
  return cudaLaunchKernelEx(&c, k_team, A);
}

}  // namespace dp
