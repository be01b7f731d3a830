// Device kernels of one propagation round (Alg. 2 of arXiv 2009.07785 with
// round-synchronous semantics) for sm_103a, plus the per-call prologue and
// epilogue.  All arithmetic that decides a bound is binary64; binary32 is
// used only in a conservative screen that proves that a nonzero cannot yield
// an accepted candidate (its binary64 candidate work is then skipped; the
// result is identical).
//
// Round structure (launched from a CUDA graph whose WHILE node repeats the
// round until k_finish clears the condition -- no host round trip):
//   k_round      one warp per slice, one lane per chunk (a block per long
//                slice where few of them have work): activities of the
//                round's chunks (Def. 1, Eq. 2a/2b, Sec. 3.4 infinity
//                counts); for whole rows also Step 2 and the binary32
//                screen, which queues the nonzeros whose candidates may be
//                accepted
//   k_combine    split rows of few pieces one per lane, rows of many pieces
//                one per warp: sums the chunk partials in a fixed order,
//                Step 2 and screen for the row
//   k_cand_split one lane per chunk of an active split row (a block per long
//                slice): queueing
//   k_cand_queue one thread per queued nonzero: the candidates (Eq. 3a/3b
//                via Eq. 5a/5b) with filtered atomics (Sec. 3.5); marks the
//                variables it updates in a dirty bitmap
//   k_finish     one warp per 8 bitmap words, per marked variable (the
//                warp together): decode the next state, crossing test
//                (Sec. 1.1, remark after Step 3), write the record the next
//                round gathers, and, when few variables changed, mark the
//                chunks that hold them: the next round skips the others (the
//                constraint marking of Alg. 1); the last block decides
//                whether to loop and whether the next round marks
// (The merge-path layout replaces the first three by the kernels of
// dp_merge.cu.)
//
// GB300 has little binary64 throughput (about 0.5 T lane-ops/s, the same for
// any number of active lanes in a warp), so binary64 work is kept lane-dense:
// the activity sums run one chunk per lane over length-sorted slices, and
// candidate formulas run 32 at a time from a per-warp work list.
#include <cuda_runtime.h>
#include <cstdint>
#include <cfloat>
#include <type_traits>

#include "dp_device.cuh"
#include "dp_internal.h"
#include "dp_round.cuh"
#include "dp_launch.h"
#include "../../include/domprop.h"

namespace dp {

// Bound candidates of one nonzero from the sides that survived the screen
// (side_candidate), applied to the next state with order-preserving 64-bit
// atomics.  Candidates are compared with the bounds at the start of the
// round (L, U).  A variable that receives a candidate is marked in the
// round's dirty bitmap; the atomics return nothing, so none of them waits
// for its answer.
__device__ __forceinline__ bool nnz_candidates(double a, int32_t j, double L, double U,
                                               uint32_t flags, unsigned sides,
                                               const RowView &rv, const Ctrl &prm,
                                               long long *keys, uint32_t *dirty) {
  const bool isint = (flags & 1u) != 0u;
  bool any = false;
  auto apply = [&](const SideCand &c) {
    if (!c.apply) return;
    if (c.upper) atomicMin(&keys[2 * (int64_t)j + 1], key_of(c.v));
    else atomicMax(&keys[2 * (int64_t)j], key_of(c.v));
    any = true;
  };
  apply(side_candidate(a, L, U, isint, (sides & 1u) != 0u, rv, prm.eps_int, prm.tau_rel,
                       prm.inf_thr));
  if (sides == 3u)  // both sides: the left-hand one too
    apply(side_candidate(a, L, U, isint, false, rv, prm.eps_int, prm.tau_rel, prm.inf_thr));
  if (any) atomicOr(&dirty[j >> 5], 1u << (j & 31));
  return any;
}

// ---------------------------------------------------------- k_cand_queue --

// Evaluates one queued nonzero.  Returns whether a candidate was applied
// (single problems: the caller sets the change flag; a set's problem's is set
// here).
template <bool kMulti, bool kCo = false>
__device__ __forceinline__ bool cand_entry_eval(const DevMatrix &M, const DevState &S,
                                                const Ctrl &prm, const CandEntry &E) {
  const uint32_t c = E.cs >> 2;
  const RowSum rs = S.rowsum[c];
  const double2 sd = S.side[c];
  const double a = ld_coef(M, E.off);
  const int32_t j = M.col[E.off];
  double L, U;
  float WU, WL;
  uint32_t fl;
  ld_rec_t<kCo>(S.rec + j, L, U, WU, WL, fl);
  RowView rv;
  rv.minfin = rs.minfin;
  rv.maxfin = rs.maxfin;
  rv.mininf = rs.mininf;
  rv.maxinf = rs.maxinf;
  rv.lhs = sd.x;
  rv.rhs = sd.y;
  rv.thr_r = rv.thr_l = f_inf();
  rv.exact = 0;
  rv.act = 1;
  const bool any = nnz_candidates(a, j, L, U, fl, E.cs & 3u, rv, prm, S.keys, S.dirty);
  if (kMulti && any) {
    int32_t *f = &S.I.changed[S.I.slot_inst[c]];
    if (__ldca(f) == 0) *f = 1;  // the flags share lines that every store would queue at
  }
  return any;
}

// Evaluates the queued nonzeros, one per thread and step, the blocks dealt out
// to the queues (block-level).  Returns whether this thread applied a candidate.
template <bool kMulti, bool kCo>
__device__ __forceinline__ bool cand_queues(const DevMatrix &M, const DevState &S,
                                            const Ctrl &prm) {
  bool any = false;
  const int nb = (int)gridDim.x;
  for (int q = (int)blockIdx.x % kQueues; q < kQueues; q += nb) {  // once, unless blocks are few
    const int32_t *n = S.qcount + q * kQueueStep;
    const int32_t cnt = kCo ? __ldcg(n) : *n;
    const CandEntry *queue = S.queue + S.qbase[q];
    const int peers = nb > q ? (nb - q + kQueues - 1) / kQueues : 1;  // blocks of this queue
    for (int64_t e = (int64_t)(blockIdx.x / kQueues) * blockDim.x + threadIdx.x; e < cnt;
         e += (int64_t)peers * blockDim.x) {
      CandEntry E;
      if (kCo) {
        const long long w = __ldcg(reinterpret_cast<const long long *>(queue + e));
        E.off = (uint32_t)w;
        E.cs = (uint32_t)((unsigned long long)w >> 32);
      } else {
        E = queue[e];
      }
      any |= cand_entry_eval<kMulti, kCo>(M, S, prm, E);
    }
  }
  return any;
}

// The grid is sized to the blocks that fit on the GPU at once.  One store per
// block sets the change flag: with one per accepted candidate the early
// rounds waited for its line.
template <bool kMulti>
__global__ void __launch_bounds__(256) k_cand_queue(DevMatrix M, DevState S) {
  const Ctrl *ctrl = S.ctrl;
  if (ctrl->err) return;
  const Ctrl prm = *ctrl;
  const bool any = cand_queues<kMulti, false>(M, S, prm);
  if (!kMulti && __syncthreads_or(any) && threadIdx.x == 0) S.ctrl->changed = 1;
}

// ------------------------------------------------------------- k_round --

// Warps per block of k_round / k_cand_split: a launch shape the autotuner
// chooses (4 or 8); the register budget per thread stays the same (24
// resident warps per SM).  24 warps with groups of four slots against 32 with
// two: 30M nonzeros of mixed rows 228 -> 210 us per round, a 2M-nonzero system
// with rows of 50,000 107 -> 70 us (its longest lanes wait for half as many
// groups); 16 x 6 and 16 x 8 are faster still on the latter and slower on the
// former (244, 268 us).
constexpr int kRoundWarpsPerSM = 24;
constexpr int kGroup = 4;         // slots per group in the activity loop

// One slice of the round (warp-level: the 32 lanes are its 32 chunks).
// kVal8: the coefficients come from the int8 copy (converted when used, so
// that the prefetched loads stay in flight).  kCo: records are loaded
// through L2 (the persistent loop).
template <bool kMulti, bool kVal8, bool kCo = false>
__device__ __forceinline__ void round_slice(const DevMatrix &M, const DevState &S, int slice,
                                            uint32_t bits) {
  constexpr int kG = kGroup;
  const Ctrl *ctrl = S.ctrl;
  const int lane = threadIdx.x & 31;
  const int64_t c = (int64_t)slice * kSliceW + lane;
  const int32_t lenf = M.chunk_len[c];
  int32_t len = lenf & kLenMask;
  int32_t row = M.chunk_row[c];
  if (!((bits >> lane) & 1u)) {  // unmarked: nothing of the row has changed
    row = -1;
    len = 0;
  }
  int32_t *inf_flag = &S.ctrl->infeasible;
  if (kMulti && row >= 0) {  // a stopped problem's rows do nothing
    const int32_t inst = S.I.slot_inst[c];
    if (S.I.done[inst]) {
      row = -1;
      len = 0;
    } else {
      inf_flag = &S.I.infeasible[inst];
    }
  }
  const int64_t sbase = M.slice_off[slice];
  const int32_t *scp = M.col + sbase;
  const int64_t vo = sbase + lane;
  const int32_t *cp = scp + lane;

  // A side's activity is needed only by rows whose side is finite (Step 2
  // and the candidates of that side); a warp skips the activity no lane
  // needs (warp-uniform: rows are ordered by side pattern when the sides
  // are known at load time).
  const double2 sd = (row >= 0) ? S.side[c] : make_double2(0.0, 0.0);  // slot order
  const bool need_min = __any_sync(kFull, row >= 0 && d_isfinite(sd.y));
  const bool need_max = __any_sync(kFull, row >= 0 && d_isfinite(sd.x));

  // ---- activities of the chunk (Def. 1, Eq. 2a/2b; Sec. 3.4) ----
  double minfin = 0.0, maxfin = 0.0;
  int32_t mininf = 0, maxinf = 0;
  Top2 t = top2_init();
  // groups of kG slots: all loads and gathers of a group are issued
  // before any is consumed, and the next group's values and columns are
  // fetched while this group's gathers are in flight; the last group's
  // missing slots are skipped (uniformly within a length-sorted slice)
  using Raw = typename std::conditional<kVal8, int, double>::type;
  auto raw = [&](int64_t off) -> Raw {
    if constexpr (kVal8) return (int)__ldcs(M.val8 + off);
    else return __ldcs(M.val + off);
  };
  auto coef = [](Raw r) -> double {
    if constexpr (kVal8) return small_int_to_double(r);
    else return r;
  };
  Raw an[kG];
  int32_t jn[kG];
#pragma unroll
  for (int u = 0; u < kG; ++u) {
    an[u] = (Raw)1;
    jn[u] = 0;
    if (u < len) {
      an[u] = raw(vo + (int64_t)u * kSliceW);
      jn[u] = __ldcs(cp + (int64_t)u * kSliceW);
    }
  }
  for (int k = 0; k < len; k += kG) {
    Raw a[kG];
    double L[kG], U[kG];
    float WU[kG], WL[kG];
    uint32_t fl[kG];
#pragma unroll
    for (int u = 0; u < kG; ++u) {
      a[u] = an[u];
      L[u] = U[u] = 0.0;
      WU[u] = WL[u] = 0.0f;
      if (k + u < len) ld_rec_t<kCo>(S.rec + jn[u], L[u], U[u], WU[u], WL[u], fl[u]);
    }
    if (k + kG < len) {
#pragma unroll
      for (int u = 0; u < kG; ++u) {
        an[u] = (Raw)1;
        jn[u] = 0;
        if (k + kG + u < len) {
          an[u] = raw(vo + (int64_t)(k + kG + u) * kSliceW);
          jn[u] = __ldcs(cp + (int64_t)(k + kG + u) * kSliceW);
        }
      }
    }
#pragma unroll
    for (int u = 0; u < kG; ++u) {
      if (k + u < len) {
        const double av = coef(a[u]);
        bool pos = d_pos(av);
        float au = absup_fast(av), ad = absdn_fast(av);
        if (need_min) {
          double bmin = pos ? L[u] : U[u];
          bool imin = d_isinf(bmin);
          mininf += imin;
          if (imin) t.kinf_min = k + u;
          minfin = fma(av, imin ? 0.0 : bmin, minfin);
          top2_add(screen_prod(au, ad, pos ? WU[u] : WL[u]), k + u, t.r1, t.r2, t.kr);
        }
        if (need_max) {
          double bmax = pos ? U[u] : L[u];
          bool imax = d_isinf(bmax);
          maxinf += imax;
          if (imax) t.kinf_max = k + u;
          maxfin = fma(av, imax ? 0.0 : bmax, maxfin);
          top2_add(screen_prod(au, ad, pos ? WL[u] : WU[u]), k + u, t.l1, t.l2, t.kl);
        }
      }
    }
  }
  const bool exact = (lenf & kExactFlag) != 0;
  if (exact) t.r1 = t.r2 = t.l1 = t.l2 = f_inf();

  if (slice < M.nslices_split) {  // warp-uniform: split chunks only
    if (row >= 0) {
      Partial p;
      p.minfin = minfin;
      p.maxfin = maxfin;
      p.mininf = mininf;
      p.maxinf = maxinf;
      p.t = t;
      p.exact = exact ? 1 : 0;
      p.pad = 0;
      S.part[c] = p;
      S.touch[M.chunk_sidx[c]] = ctrl->round + 1;
    }
    return;
  }

  // ---- whole rows: Step 2, screen, candidates ----
  RowView rv;
  rv.minfin = minfin;
  rv.maxfin = maxfin;
  rv.mininf = mininf;
  rv.maxinf = maxinf;
  rv.exact = exact ? 1 : 0;
  rv.act = 0;
  rv.thr_r = rv.thr_l = f_inf();
  if (row >= 0) {
    rv.lhs = sd.x;
    rv.rhs = sd.y;
    row_sides(rv, t.r1, t.l1, ctrl->eps_feas, inf_flag);
  } else {
    rv.lhs = rv.rhs = 0.0;
  }
  warp_enqueue<kSliceW, kCo>(rv, t, mininf, maxinf, len, c, sbase + lane, M, M.col, S);
}

// A slice of whole rows of at most kShortRow nonzeros (warp-level): the
// lanes keep their rows' screen values in registers, so the survivors are
// queued without a second pass over the nonzeros, and one-sided slices (most)
// run code for one side.  30M nonzeros of mixed rows, 97% of the rows this
// short: 210 -> 189 us per round.  Longer rows would need more registers than
// 24 resident warps leave; in a kernel of its own, before, behind or beside
// k_round in the graph, the same code made the round slower (265 us), since
// nothing then fills the SMs while the long slices finish.
template <int kSides>
__device__ __forceinline__ void short_rows(const DevMatrix &M, const DevState &S, int64_t c,
                                           int64_t elem0, int32_t len, int32_t row, bool exact,
                                           double2 sd, bool right, int32_t *inf_flag) {
  ShortAct<kSides, kShortRow> r;
  short_activity<kSides, kShortRow>(
      M, elem0, len, right,
      [&](int32_t j, double &L, double &U, float &WU, float &WL) {
        uint32_t fl;
        ld_rec(S.rec + j, L, U, WU, WL, fl);
      },
      r);
  constexpr int kR = 0, kL = kSides - 1;  // one side: both names are its index
  const bool use_r = kSides == 2 || right, use_l = kSides == 2 || !right;
  RowView rv;
  rv.minfin = use_r ? r.fin[kR] : 0.0;
  rv.maxfin = use_l ? r.fin[kL] : 0.0;
  rv.mininf = use_r ? r.ninf[kR] : 0;
  rv.maxinf = use_l ? r.ninf[kL] : 0;
  rv.exact = exact ? 1 : 0;
  rv.act = 0;
  rv.thr_r = rv.thr_l = f_inf();
  rv.lhs = sd.x;
  rv.rhs = sd.y;
  uint32_t mr = 0u, ml = 0u;
  if (row >= 0) {
    row_sides(rv, !use_r ? -f_inf() : (exact ? f_inf() : short_max(r.t[kR])),
              !use_l ? -f_inf() : (exact ? f_inf() : short_max(r.t[kL])), S.ctrl->eps_feas,
              inf_flag);
    if (rv.act) {
      if (use_r)
        mr = short_survivors(r.t[kR], len, d_isfinite(rv.rhs), rv.mininf, r.kinf[kR], rv.thr_r,
                             exact);
      if (use_l)
        ml = short_survivors(r.t[kL], len, d_isfinite(rv.lhs), rv.maxinf, r.kinf[kL], rv.thr_l,
                             exact);
    }
  }
  uint32_t m = mr | ml;
  uint32_t pos = warp_reserve<4>(__popc(m), c, S);
  if (m == 0u) return;
  RowSum rs;
  rs.minfin = rv.minfin;
  rs.maxfin = rv.maxfin;
  rs.mininf = rv.mininf;
  rs.maxinf = rv.maxinf;
  S.rowsum[c] = rs;
  for (; m != 0u; m &= m - 1u, ++pos) {
    const int k = __ffs(m) - 1;
    CandEntry e;
    e.off = (uint32_t)(elem0 + k * kSliceW);
    e.cs = ((uint32_t)c << 2) | ((mr >> k) & 1u) | (((ml >> k) & 1u) << 1);
    S.queue[pos] = e;
  }
}

template <bool kMulti>
__device__ __forceinline__ void short_slice(const DevMatrix &M, const DevState &S, int slice,
                                            uint32_t bits) {
  const int lane = threadIdx.x & 31;
  const int64_t c = (int64_t)slice * kSliceW + lane;
  const int32_t lenf = M.chunk_len[c];
  int32_t len = lenf & kLenMask;
  int32_t row = M.chunk_row[c];
  if (!((bits >> lane) & 1u)) {  // unmarked: nothing of the row has changed
    row = -1;
    len = 0;
  }
  int32_t *inf_flag = &S.ctrl->infeasible;
  if (kMulti && row >= 0) {  // a stopped problem's rows do nothing
    const int32_t inst = S.I.slot_inst[c];
    if (S.I.done[inst]) {
      row = -1;
      len = 0;
    } else {
      inf_flag = &S.I.infeasible[inst];
    }
  }
  const double2 sd = (row >= 0) ? S.side[c] : make_double2(0.0, 0.0);
  const bool need_min = __any_sync(kFull, row >= 0 && d_isfinite(sd.y));
  const bool need_max = __any_sync(kFull, row >= 0 && d_isfinite(sd.x));
  const int64_t elem0 = M.slice_off[slice] + lane;
  const bool exact = (lenf & kExactFlag) != 0;
  if (need_min && need_max)
    short_rows<2>(M, S, c, elem0, len, row, exact, sd, true, inf_flag);
  else
    short_rows<1>(M, S, c, elem0, len, row, exact, sd, need_min, inf_flag);
}

// What a lane knows about its chunk before it reads any nonzero.
struct ChunkHead {
  int64_t c;      // chunk slot
  int32_t len, row;  // 0 and -1 for padding, unmarked chunks, a stopped problem's rows
  bool exact;     // the row skips the binary32 screen
  double2 sd;     // {lhs, rhs}
  bool need_min, need_max;  // warp-uniform: some lane's row needs that activity
  int32_t *inf_flag;
};

// A side's activity is needed only by rows whose side is finite (Step 2 and
// the candidates of that side); a warp skips the activity no lane needs
// (warp-uniform: rows are ordered by side pattern when the sides are known
// at load time).
// `bits`: the chunks of the slice to process.
template <bool kMulti>
__device__ __forceinline__ ChunkHead chunk_head(const DevMatrix &M, const DevState &S, int slice,
                                                uint32_t bits) {
  ChunkHead h;
  h.c = (int64_t)slice * kSliceW + (threadIdx.x & 31);
  const int32_t lenf = M.chunk_len[h.c];
  h.len = lenf & kLenMask;
  h.exact = (lenf & kExactFlag) != 0;
  h.row = M.chunk_row[h.c];
  if (!((bits >> (threadIdx.x & 31)) & 1u)) {
    h.row = -1;
    h.len = 0;
  }
  h.inf_flag = &S.ctrl->infeasible;
  if (kMulti && h.row >= 0) {  // a stopped problem's rows do nothing
    const int32_t inst = S.I.slot_inst[h.c];
    if (S.I.done[inst]) {
      h.row = -1;
      h.len = 0;
    } else {
      h.inf_flag = &S.I.infeasible[inst];
    }
  }
  h.sd = (h.row >= 0) ? S.side[h.c] : make_double2(0.0, 0.0);  // slot order
  h.need_min = __any_sync(kFull, h.row >= 0 && d_isfinite(h.sd.y));
  h.need_max = __any_sync(kFull, h.row >= 0 && d_isfinite(h.sd.x));
  return h;
}

// A chunk's infinity counts and screen top-2, lane-level; the finite sums
// are kept apart (round_slice adds them here, team_slice in its chain).
struct ChunkAcc {
  int32_t mininf, maxinf;
  Top2 t;
};

// One nonzero's contribution apart from the finite sums; returns the
// bounds those sums use (0 in the place of an infinite one).
__device__ __forceinline__ void acc_nnz(double av, double L, double U, float WU, float WL, int k,
                                        bool need_min, bool need_max, ChunkAcc &r, double &bmin,
                                        double &bmax) {
  const bool pos = d_pos(av);
  const float au = absup_fast(av), ad = absdn_fast(av);
  if (need_min) {
    bmin = pos ? L : U;
    const bool inf = d_isinf(bmin);
    r.mininf += inf;
    if (inf) r.t.kinf_min = k;
    bmin = inf ? 0.0 : bmin;
    top2_add(screen_prod(au, ad, pos ? WU : WL), k, r.t.r1, r.t.r2, r.t.kr);
  }
  if (need_max) {
    bmax = pos ? U : L;
    const bool inf = d_isinf(bmax);
    r.maxinf += inf;
    if (inf) r.t.kinf_max = k;
    bmax = inf ? 0.0 : bmax;
    top2_add(screen_prod(au, ad, pos ? WL : WU), k, r.t.l1, r.t.l2, r.t.kl);
  }
}

// The coefficient stream: binary64, or the int8 copy (converted when used,
// so that the prefetched loads stay in flight).
template <bool kVal8>
using Raw = typename std::conditional<kVal8, int, double>::type;
template <bool kVal8>
__device__ __forceinline__ double coef_of(Raw<kVal8> r) {
  if constexpr (kVal8) return small_int_to_double(r);
  else return r;
}

__device__ __forceinline__ void put_partial(const ChunkHead &h, const ChunkAcc &r, double minfin,
                                            double maxfin, const DevMatrix &M,
                                            const DevState &S) {
  Partial p;
  p.minfin = minfin;
  p.maxfin = maxfin;
  p.mininf = r.mininf;
  p.maxinf = r.maxinf;
  p.t = r.t;
  p.exact = h.exact ? 1 : 0;
  p.pad = 0;
  S.part[h.c] = p;
  S.touch[M.chunk_sidx[h.c]] = S.ctrl->round + 1;
}

// Step 2 and the screen thresholds of the lane's whole row.
__device__ __forceinline__ RowView whole_row(const ChunkHead &h, const ChunkAcc &r, double minfin,
                                             double maxfin, double eps_feas) {
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
  if (h.row >= 0) row_sides(rv, r.t.r1, r.t.l1, eps_feas, h.inf_flag);
  return rv;
}

// ---- long slices: one slice per block ----
//
// A lane of round_slice spends about 0.17 us per slot on dependent
// instructions alone (plus the latency of each group's gathers), so a slice
// of 256 slots takes 70-110 us however empty the GPU is, and on a matrix
// with any long row that is what the round waits for (2M nonzeros with rows of
// 20,000 to 50,000: 70 -> 40 us per round; 6M with rows of up to 100,000: 99 ->
// 61).  A block costs 1.5 times the warp-time per slice, so it pays while the
// blocks' slices are few (30M nonzeros, 15 long slices per SM: 210 -> 340).  Here the block's
// warps take U consecutive slots each, so that loads, gathers and the screen
// run side by side; the bounds go through shared memory to one warp per side
// that adds them slot by slot.  The finite sums thus stay one FMA chain per
// row in CSR order, the same bits as round_slice, and the chain (about 64
// clocks per slot: the binary64 pipe) is all that remains serial.
constexpr int kTeamU = 2;            // slots per warp and step
constexpr int kTeamBlocksPerSM = 4;  // long slices per SM up to which a block takes each

template <int kWarps>
struct TeamBuf {
  static constexpr int kStep = kWarps * kTeamU;
  union {
    double b[2][2][kStep][kSliceW];      // [side][buffer][slot][lane] bounds of a step
    ChunkAcc part[kWarps][kSliceW];      // the warps' shares of the chunks
  };
  double fin[2][kSliceW];
  RowView rv[kSliceW];
  int32_t len[kSliceW];  // slots to re-read of each chunk
};

template <bool kMulti, int kWarps, bool kVal8>
__device__ __forceinline__ void team_slice(const DevMatrix &M, const DevState &S, int slice,
                                           uint32_t bits, TeamBuf<kWarps> &sb) {
  constexpr int U = kTeamU, kStep = TeamBuf<kWarps>::kStep;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const ChunkHead h = chunk_head<kMulti>(M, S, slice, bits);
  const int32_t len = h.len;
  const int maxlen = __reduce_max_sync(kFull, len);  // the same in every warp
  const int64_t vo = M.slice_off[slice] + lane;
  const int32_t *cp = M.col + vo;
  const bool need_min = h.need_min, need_max = h.need_max;
  // the warps that add up the sides: on different binary64 pipes, and not
  // the same ones in every block
  const int wmin = blockIdx.x % kWarps, wmax = (blockIdx.x + 1) % kWarps;
  double fin = 0.0;
  ChunkAcc r;
  r.mininf = r.maxinf = 0;
  r.t = top2_init();
  Raw<kVal8> an[U];
  int32_t jn[U];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      an[u] = (Raw<kVal8>)1;
      jn[u] = 0;
      if (k0 + u < len) {
        if constexpr (kVal8) an[u] = (int)__ldg(M.val8 + vo + (int64_t)(k0 + u) * kSliceW);
        else an[u] = __ldg(M.val + vo + (int64_t)(k0 + u) * kSliceW);
        jn[u] = __ldg(cp + (int64_t)(k0 + u) * kSliceW);
      }
    }
  };
  // adds the staged step that began at slot s0 (its coefficients are in L1)
  auto chain = [&](int s0, int side) {
    const double(*bb)[kSliceW] = sb.b[side][(s0 / kStep) & 1];
    for (int q = 0; q < kStep; q += 4) {
      Raw<kVal8> a[4];
      double b[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        a[u] = (Raw<kVal8>)1;
        b[u] = 0.0;
        if (s0 + q + u < len) {
          if constexpr (kVal8) a[u] = (int)__ldg(M.val8 + vo + (int64_t)(s0 + q + u) * kSliceW);
          else a[u] = __ldg(M.val + vo + (int64_t)(s0 + q + u) * kSliceW);
          b[u] = bb[q + u][lane];
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (s0 + q + u < len) fin = fma(coef_of<kVal8>(a[u]), b[u], fin);
    }
  };
  fetch(warp * U);
  for (int s = 0; s < maxlen; s += kStep) {
    const int k = s + warp * U;
    Raw<kVal8> a[U];
    double L[U], Ub[U];
    float WU[U], WL[U];
    uint32_t fl[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      a[u] = an[u];
      L[u] = Ub[u] = 0.0;
      WU[u] = WL[u] = 0.0f;
      if (k + u < len) ld_rec(S.rec + jn[u], L[u], Ub[u], WU[u], WL[u], fl[u]);
    }
    fetch(k + kStep);
    if (s > 0 && need_min && warp == wmin) chain(s - kStep, 0);
    if (s > 0 && need_max && warp == wmax) chain(s - kStep, 1);
    const int buf = (s / kStep) & 1;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (k + u < len) {
        double bmin, bmax;
        acc_nnz(coef_of<kVal8>(a[u]), L[u], Ub[u], WU[u], WL[u], k + u, need_min, need_max, r,
                bmin, bmax);
        if (need_min) sb.b[0][buf][warp * U + u][lane] = bmin;
        if (need_max) sb.b[1][buf][warp * U + u][lane] = bmax;
      }
    }
    __syncthreads();  // the step is staged, and the step before it is added
  }
  if (maxlen > 0) {
    const int last = (maxlen - 1) / kStep * kStep;
    if (need_min && warp == wmin) chain(last, 0);
    if (need_max && warp == wmax) chain(last, 1);
    __syncthreads();  // the staging is free for the warps' parts
  }
  sb.part[warp][lane] = r;
  if (warp == wmin) sb.fin[0][lane] = need_min ? fin : 0.0;
  if (kWarps > 1 && warp == wmax) sb.fin[1][lane] = need_max ? fin : 0.0;
  __syncthreads();
  if (warp == 0) {
#pragma unroll 1
    for (int w = 1; w < kWarps; ++w) {
      const ChunkAcc q = sb.part[w][lane];
      if (q.mininf > 0) r.t.kinf_min = q.t.kinf_min;
      if (q.maxinf > 0) r.t.kinf_max = q.t.kinf_max;
      r.mininf += q.mininf;
      r.maxinf += q.maxinf;
      top2_merge(q.t.r1, q.t.r2, q.t.kr, r.t.r1, r.t.r2, r.t.kr);
      top2_merge(q.t.l1, q.t.l2, q.t.kl, r.t.l1, r.t.l2, r.t.kl);
    }
    if (h.exact) r.t.r1 = r.t.r2 = r.t.l1 = r.t.l2 = f_inf();
    const double minfin = sb.fin[0][lane], maxfin = sb.fin[1][lane];
    if (slice < M.nslices_split) {
      if (h.row >= 0) put_partial(h, r, minfin, maxfin, M, S);
    } else {
      const RowView rv = whole_row(h, r, minfin, maxfin, S.ctrl->eps_feas);
      const bool full =
          enqueue_named<kSliceW>(rv, r.t, r.mininf, r.maxinf, h.c, vo, S);
      sb.rv[lane] = rv;
      sb.len[lane] = full ? len : 0;
    }
  }
  if (slice < M.nslices_split) return;  // block-uniform
  __syncthreads();
  // the re-read of rows with several survivors, shared by the warps
  const int32_t rlen = sb.len[lane];
  if (__ballot_sync(kFull, rlen > 0) == 0u) return;
  const RowView rv = sb.rv[lane];
  enqueue_reread<kSliceW, false>(rv, rlen, warp * 4, kWarps * 4, h.c, vo, M, M.col, S);
}

// ---- one chunk per warp ----
//
// Late rounds mark a few chunks only.  A long one then goes to a warp of its
// own: the lanes gather 32 slots side by side, and the chain runs over
// shuffled values (lanes below 16 add up the minimum activity, the others
// the maximum): the same FMA chain in CSR order, 64 clocks per slot, where a
// lane alone takes about 310 (256 slots: 12-20 us instead of 75).
__device__ __forceinline__ void coop_activity(const DevMatrix &M, const VarRec *rec,
                                              int64_t elem0, int32_t len, bool need_min,
                                              bool need_max, ChunkAcc &r, double &minfin,
                                              double &maxfin) {
  const int lane = threadIdx.x & 31;
  double fin = 0.0;
  r.mininf = r.maxinf = 0;
  r.t = top2_init();
  for (int t0 = 0; t0 < len; t0 += 128) {
    double a[4], bmin[4], bmax[4];
    int32_t j[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int k = t0 + 32 * u + lane;
      a[u] = 1.0;
      j[u] = 0;
      bmin[u] = bmax[u] = 0.0;
      if (k < len) {
        a[u] = ld_coef(M, elem0 + (int64_t)k * kSliceW);
        j[u] = M.col[elem0 + (int64_t)k * kSliceW];
      }
    }
    double L[4], U[4];
    float WU[4], WL[4];
    uint32_t fl;
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (t0 + 32 * u + lane < len) ld_rec(rec + j[u], L[u], U[u], WU[u], WL[u], fl);
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (t0 + 32 * u + lane < len)
        acc_nnz(a[u], L[u], U[u], WU[u], WL[u], t0 + 32 * u + lane, need_min, need_max, r,
                bmin[u], bmax[u]);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int n = min(32, len - t0 - 32 * u);
      for (int i = 0; i < n; ++i) {  // warp-uniform
        const double av = __shfl_sync(kFull, a[u], i);
        const double bn = __shfl_sync(kFull, bmin[u], i), bx = __shfl_sync(kFull, bmax[u], i);
        fin = fma(av, lane < 16 ? bn : bx, fin);
      }
    }
  }
  minfin = need_min ? __shfl_sync(kFull, fin, 0) : 0.0;
  maxfin = need_max ? __shfl_sync(kFull, fin, 16) : 0.0;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const int32_t mi = __shfl_xor_sync(kFull, r.mininf, o), xi = __shfl_xor_sync(kFull, r.maxinf, o);
    const int32_t km = __shfl_xor_sync(kFull, r.t.kinf_min, o);
    const int32_t kx = __shfl_xor_sync(kFull, r.t.kinf_max, o);
    if (r.mininf == 0) r.t.kinf_min = km;
    if (r.maxinf == 0) r.t.kinf_max = kx;
    r.mininf += mi;
    r.maxinf += xi;
    const float r1 = __shfl_xor_sync(kFull, r.t.r1, o), r2 = __shfl_xor_sync(kFull, r.t.r2, o);
    const float l1 = __shfl_xor_sync(kFull, r.t.l1, o), l2 = __shfl_xor_sync(kFull, r.t.l2, o);
    const int32_t kr = __shfl_xor_sync(kFull, r.t.kr, o), kl = __shfl_xor_sync(kFull, r.t.kl, o);
    top2_merge(r1, r2, kr, r.t.r1, r.t.r2, r.t.kr);
    top2_merge(l1, l2, kl, r.t.l1, r.t.l2, r.t.kl);
  }
}

// A marked chunk of a long slice (warp-level).
template <bool kMulti>
__device__ __forceinline__ void coop_chunk(const DevMatrix &M, const DevState &S, int slice,
                                           int which) {
  const int lane = threadIdx.x & 31;
  // every lane looks at the same chunk
  ChunkHead h;
  h.c = (int64_t)slice * kSliceW + which;
  const int32_t lenf = M.chunk_len[h.c];
  h.len = lenf & kLenMask;
  h.exact = (lenf & kExactFlag) != 0;
  h.row = M.chunk_row[h.c];
  if (h.row < 0) return;
  h.inf_flag = &S.ctrl->infeasible;
  if (kMulti) {
    const int32_t inst = S.I.slot_inst[h.c];
    if (S.I.done[inst]) return;
    h.inf_flag = &S.I.infeasible[inst];
  }
  h.sd = S.side[h.c];
  const int64_t elem0 = M.slice_off[slice] + which;
  ChunkAcc r;
  double minfin, maxfin;
  coop_activity(M, S.rec, elem0, h.len, d_isfinite(h.sd.y), d_isfinite(h.sd.x), r,
                              minfin, maxfin);
  if (h.exact) r.t.r1 = r.t.r2 = r.t.l1 = r.t.l2 = f_inf();
  if (slice < M.nslices_split) {
    if (lane == 0) put_partial(h, r, minfin, maxfin, M, S);
    return;
  }
  RowView rv = whole_row(h, r, minfin, maxfin, S.ctrl->eps_feas);
  const bool act = rv.act != 0;
  if (lane != 0) rv.act = 0;  // one lane speaks for the row
  bool full = enqueue_named<kSliceW>(rv, r.t, r.mininf, r.maxinf, h.c, elem0, S);
  full = __shfl_sync(kFull, full, 0);
  if (!act || !full) return;
  for (int k0 = 0; k0 < h.len; k0 += 32) {  // the re-read, a slot per lane
    const int k = k0 + lane;
    unsigned sides = 0u;
    if (k < h.len) {
      double L, U;
      float WU, WL;
      uint32_t fl;
      const double a = ld_coef(M, elem0 + (int64_t)k * kSliceW);
      ld_rec(S.rec + M.col[elem0 + (int64_t)k * kSliceW], L, U, WU, WL, fl);
      sides = nnz_sides(a, L, U, WU, WL, rv);
    }
    warp_push(sides != 0u, elem0 + (int64_t)k * kSliceW, h.c, sides, S);
  }
}

// The q-th slice of a round, the long ones first.
__device__ __forceinline__ int nth_slice(const DevMatrix &M, int q) {
  if (M.order) return M.order[q];
  const int nlong = M.long_split + M.long_whole;
  if (q < nlong) return q < M.long_split ? q : M.nslices_split + (q - M.long_split);
  q -= nlong;
  const int rest = M.nslices_split - M.long_split;  // split slices that are not long
  return q < rest ? M.long_split + q : M.nslices_split + M.long_whole + (q - rest);
}

// The chunks of a slice to process this round (warp-uniform), and the
// slice's mask cleared for the next one: every chunk in the first round and
// after a round that changed too many variables to mark their rows one by
// one, else those with a variable that changed in the previous round.
// Skipping the others is exact (the constraint marking of Alg. 1, Sec. 2.1):
// their activities, hence their candidates, are those of the round that
// processed them last, applied or rejected then against bounds that have
// only tightened since.
__device__ __forceinline__ uint32_t take_mask(const DevState &S, int slice, bool all) {
  uint32_t m = 0u;
  if ((threadIdx.x & 31) == 0) {
    m = S.mask[slice];
    if (m != 0u) S.mask[slice] = 0u;
  }
  return all ? kFull : __shfl_sync(kFull, m, 0);
}

// The nlong long slices first, the others by a warp each.  A block takes a
// long slice when there are few of them (`few`) or very few chunks are marked
// (30M nonzeros, 15 long slices per SM, 0.05% of the variables changed: 84 ->
// 49 us; with 1% changed the blocks are slower, 171 -> 321 us); else it takes
// kRoundWarps of them, and the blocks left over return.
template <bool kMulti, int kRoundWarps, bool kVal8>
__global__ void __launch_bounds__(kRoundWarps * 32, kRoundWarpsPerSM / kRoundWarps)
k_round(DevMatrix M, DevState S, int few) {
  __shared__ TeamBuf<kRoundWarps> sb;
  __shared__ uint32_t s_bits;
  if (S.ctrl->err) return;
  const bool all = S.ctrl->all_active != 0;
  const int b = (int)blockIdx.x, warp = threadIdx.x >> 5;
  if (b < M.nlong && (few || S.ctrl->sparse)) {
    const int slice = nth_slice(M, b);
    if (warp == 0) {
      const uint32_t m = take_mask(S, slice, all);
      if (threadIdx.x == 0) s_bits = m;
    }
    __syncthreads();
    uint32_t m = s_bits;
    if (__popc(m) <= kRoundWarps) {  // few chunks: one per warp
      for (int at = 0; m != 0u; m &= m - 1u, ++at)
        if (at == warp) coop_chunk<kMulti>(M, S, slice, __ffs(m) - 1);
    } else {
      team_slice<kMulti, kRoundWarps, kVal8>(M, S, slice, m, sb);
    }
    return;
  }
  const int q = b < M.nlong ? b * kRoundWarps + warp
                            : M.nlong + (b - M.nlong) * kRoundWarps + warp;
  if (q >= (b < M.nlong ? M.nlong : M.nslices)) return;  // warp-uniform
  const int slice = nth_slice(M, q);
  const uint32_t bits = take_mask(S, slice, all);
  if (bits == 0u) return;
  if (!kVal8 && q >= M.short0) short_slice<kMulti>(M, S, slice, bits);
  else round_slice<kMulti, kVal8>(M, S, slice, bits);
}

// ------------------------------------------------------------- k_floor --
//
// The memory access pattern of k_round's activity pass alone, on the same
// layout and in the same launch shape: every slot's value and column
// streamed, every nonzero's 32-byte record gathered, no arithmetic beyond an
// integer fold that keeps the loads alive.  Its time is the floor that the
// round kernel's memory traffic sets on this matrix (a measurement, not part
// of propagation).
template <int kRoundWarps>
__global__ void __launch_bounds__(kRoundWarps * 32, kRoundWarpsPerSM / kRoundWarps)
k_floor(DevMatrix M, DevState S, int teams, unsigned *sink) {
  const int warp = threadIdx.x >> 5;
  const bool team = (int)blockIdx.x < teams;  // its warps share the slice's slots
  const int q = team ? (int)blockIdx.x
                     : teams + ((int)blockIdx.x - teams) * kRoundWarps + warp;
  if (q >= M.nslices) return;
  const int slice = nth_slice(M, q);
  const int kbeg = team ? warp * kGroup : 0, kstep = team ? kRoundWarps * kGroup : kGroup;
  const int lane = threadIdx.x & 31;
  const int64_t c = (int64_t)slice * kSliceW + lane;
  const int32_t len = M.chunk_len[c] & kLenMask;
  const int64_t vo = M.slice_off[slice] + lane;
  unsigned acc = 0u;
  for (int k = kbeg; k < len; k += kstep) {
    double a[kGroup];
    int32_t j[kGroup];
#pragma unroll
    for (int u = 0; u < kGroup; ++u) {
      a[u] = 0.0;
      j[u] = 0;
      if (k + u < len) {
        a[u] = __ldcs(M.val + vo + (int64_t)(k + u) * kSliceW);
        j[u] = __ldcs(M.col + vo + (int64_t)(k + u) * kSliceW);
      }
    }
#pragma unroll
    for (int u = 0; u < kGroup; ++u) {
      if (k + u < len) {
        double L, U;
        float WU, WL;
        uint32_t fl;
        ld_rec(S.rec + j[u], L, U, WU, WL, fl);
        acc ^= (unsigned)__double_as_longlong(L) ^ (unsigned)__double_as_longlong(a[u]) ^
               __float_as_uint(WU) ^ fl;
      }
    }
  }
  if (acc == 0x9E3779B9u) *sink = acc;  // practically never: keeps the loads
}

// Slices that a block takes each: the long ones, when they are few.
static int team_blocks(const DevMatrix &M, int num_sms) {
  return M.nlong <= kTeamBlocksPerSM * num_sms ? M.nlong : 0;
}

cudaError_t launch_access_floor(const DevMatrix &M, const DevState &S, unsigned *sink,
                                int num_sms, cudaStream_t st) {
  if (M.layout != kLayoutEll) return cudaErrorInvalidValue;
  const int w = M.round_warps == 4 ? 4 : 8;
  const int teams = team_blocks(M, num_sms);
  int nb = teams + (M.nslices - teams + w - 1) / w;
  if (nb < 1) nb = 1;
  if (w == 4) k_floor<4><<<nb, 4 * 32, 0, st>>>(M, S, teams, sink);
  else k_floor<8><<<nb, 8 * 32, 0, st>>>(M, S, teams, sink);
  return cudaGetLastError();
}

// ------------------------------------------------------------ k_combine --

constexpr int kCombineWarps = 8;
constexpr int kCombineShort = 4;  // rows with at most this many pieces: their own lane

// Running sums of a split row's pieces.
struct RowAcc {
  double mnf, mxf;
  int32_t mni, mxi, ex;
  float Tr, Tl;
};

__device__ __forceinline__ void acc_init(RowAcc &a) {
  a.mnf = a.mxf = 0.0;
  a.mni = a.mxi = a.ex = 0;
  a.Tr = a.Tl = -f_inf();
}

__device__ __forceinline__ void acc_add(RowAcc &a, const Partial &p) {
  a.mnf += p.minfin;
  a.mxf += p.maxfin;
  a.mni += p.mininf;
  a.mxi += p.maxinf;
  a.Tr = fmaxf(a.Tr, p.t.r1);
  a.Tl = fmaxf(a.Tl, p.t.l1);
  a.ex |= p.exact;
}

// Step 2 and the screen thresholds of split row w from its sums (thread-level).
__device__ __forceinline__ void combine_commit(const DevMatrix &M, const DevState &S, int64_t w,
                                               RowAcc &a, int32_t *inf_flag) {
  const int32_t row = M.split_row[w];
  RowView rv;
  rv.minfin = a.mnf;
  rv.maxfin = a.mxf;
  rv.mininf = a.mni;
  rv.maxinf = a.mxi;
  rv.lhs = S.lhs[row];
  rv.rhs = S.rhs[row];
  rv.exact = a.ex;
  if (a.ex) a.Tr = a.Tl = f_inf();
  row_sides(rv, a.Tr, a.Tl, S.ctrl->eps_feas, inf_flag);
  RowTot rt;
  rt.minfin = a.mnf;
  rt.maxfin = a.mxf;
  rt.mininf = a.mni;
  rt.maxinf = a.mxi;
  rt.thr_r = rv.thr_r;
  rt.thr_l = rv.thr_l;
  rt.active = rv.act;
  rt.row = row;
  S.rowtot[w] = rt;
}

// Warp w of the split-row pass (warp-level, all 32 lanes): rows [32w,
// 32w + 32) of at most kCombineShort pieces are summed each by its own lane
// in piece order; row w, if it has more pieces, by the whole warp, lanes
// strided over its pieces and then a fixed butterfly (reproducible, and the
// same in every lane).  Which of the two sums a row depends only on its
// piece count, and every row is summed once.
template <bool kMulti>
__device__ __forceinline__ void combine_rows(const DevMatrix &M, const DevState &S, int64_t w) {
  const int lane = threadIdx.x & 31;
  auto flag_of = [&](int32_t first_piece) -> int32_t * {
    return kMulti ? &S.I.infeasible[S.I.slot_inst[M.split_cidx[first_piece]]]
                  : &S.ctrl->infeasible;
  };
  // a row none of whose pieces was recomputed this round has no new candidates
  const int32_t now = S.ctrl->round + 1;
  auto stopped = [&](int32_t first_piece) {  // a stopped problem: no candidates
    return kMulti && S.I.done[S.I.slot_inst[M.split_cidx[first_piece]]];
  };
  // short rows, one per lane
  const int64_t r = w * 32 + lane;
  if (r < M.nsplit_rows) {
    const int32_t cb = M.split_cbeg[r], ce = M.split_cbeg[r + 1];
    if (ce - cb <= kCombineShort) {
      if (stopped(cb) || S.touch[r] != now) {
        S.rowtot[r].active = 0;
      } else {
        RowAcc a;
        acc_init(a);
        Partial p[kCombineShort];
#pragma unroll
        for (int u = 0; u < kCombineShort; ++u)
          if (cb + u < ce) p[u] = S.part[M.split_cidx[cb + u]];
#pragma unroll
        for (int u = 0; u < kCombineShort; ++u)
          if (cb + u < ce) acc_add(a, p[u]);
        combine_commit(M, S, r, a, flag_of(cb));
      }
    }
  }
  // row w if it has many pieces (warp-uniform)
  const int32_t b = M.split_cbeg[w], e = M.split_cbeg[w + 1];
  if (e - b <= kCombineShort) return;
  if (stopped(b) || S.touch[w] != now) {
    if (lane == 0) S.rowtot[w].active = 0;
    return;
  }
  RowAcc a;
  acc_init(a);
  // each lane sums its pieces in order; the loads of four pieces are issued
  // before they are consumed
  int32_t q = b + lane;
  for (; q + 3 * kSliceW < e; q += 4 * kSliceW) {
    int32_t ci[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) ci[u] = M.split_cidx[q + u * kSliceW];
    Partial p[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) p[u] = S.part[ci[u]];
#pragma unroll
    for (int u = 0; u < 4; ++u) acc_add(a, p[u]);
  }
  for (; q < e; q += kSliceW) acc_add(a, S.part[M.split_cidx[q]]);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    a.mnf += __shfl_xor_sync(kFull, a.mnf, off);
    a.mxf += __shfl_xor_sync(kFull, a.mxf, off);
    a.mni += __shfl_xor_sync(kFull, a.mni, off);
    a.mxi += __shfl_xor_sync(kFull, a.mxi, off);
    a.Tr = fmaxf(a.Tr, __shfl_xor_sync(kFull, a.Tr, off));
    a.Tl = fmaxf(a.Tl, __shfl_xor_sync(kFull, a.Tl, off));
    a.ex |= __shfl_xor_sync(kFull, a.ex, off);
  }
  if (lane == 0) combine_commit(M, S, w, a, flag_of(b));
}

template <bool kMulti>
__global__ void __launch_bounds__(kCombineWarps * 32)
k_combine(DevMatrix M, DevState S) {
  if (S.ctrl->err) return;
  const int64_t w = blockIdx.x * (int64_t)kCombineWarps + (threadIdx.x >> 5);
  if (w >= M.nsplit_rows) return;  // warp-uniform
  combine_rows<kMulti>(M, S, w);
}

// --------------------------------------------------------- k_cand_split --

// The state of the active split rows' chunks of one slice: the row's sums
// and thresholds, the chunk's top-2 (lane-level).
struct SplitChunk {
  RowView rv;
  Top2 t;
  int32_t len, mininf, maxinf;
};

__device__ __forceinline__ SplitChunk split_chunk(const DevMatrix &M, const DevState &S,
                                                  int64_t c) {
  SplitChunk x;
  const int32_t sidx = M.chunk_sidx[c];
  x.rv.act = 0;
  x.rv.exact = 0;
  x.rv.mininf = x.rv.maxinf = 0;
  x.rv.minfin = x.rv.maxfin = x.rv.lhs = x.rv.rhs = 0.0;
  x.rv.thr_r = x.rv.thr_l = f_inf();
  x.t = top2_init();
  x.len = x.mininf = x.maxinf = 0;
  if (sidx >= 0) {
    const RowTot rt = S.rowtot[sidx];
    if (rt.active) {
      const Partial p = S.part[c];
      const int32_t lenf = M.chunk_len[c];
      x.len = lenf & kLenMask;
      x.rv.minfin = rt.minfin;
      x.rv.maxfin = rt.maxfin;
      x.rv.mininf = rt.mininf;
      x.rv.maxinf = rt.maxinf;
      x.rv.thr_r = rt.thr_r;
      x.rv.thr_l = rt.thr_l;
      x.rv.lhs = S.lhs[rt.row];
      x.rv.rhs = S.rhs[rt.row];
      x.rv.exact = (lenf & kExactFlag) ? 1 : 0;
      x.rv.act = 1;
      x.t = p.t;
      x.mininf = p.mininf;
      x.maxinf = p.maxinf;
    }
  }
  return x;
}

// Candidates of the active split rows' chunks of one slice (warp-level).
template <bool kCo = false>
__device__ __forceinline__ void cand_split_slice(const DevMatrix &M, const DevState &S,
                                                 int slice) {
  const int lane = threadIdx.x & 31;
  const int64_t c = (int64_t)slice * kSliceW + lane;
  const SplitChunk x = split_chunk(M, S, c);
  warp_enqueue<kSliceW, kCo>(x.rv, x.t, x.mininf, x.maxinf, x.len, c, M.slice_off[slice] + lane,
                             M, M.col, S);
}

// A block per long slice (its warps share the re-read, which one lane's walk
// made the longest part of early rounds: 30M nonzeros 42 -> 15 us per round), a
// warp per other one.
template <int kRoundWarps>
__global__ void __launch_bounds__(kRoundWarps * 32)
k_cand_split(DevMatrix M, DevState S) {
  if (S.ctrl->err) return;
  __shared__ int32_t s_len[kSliceW];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (blockIdx.x >= M.long_split) {
    const int slice = M.long_split + ((int)blockIdx.x - M.long_split) * kRoundWarps + warp;
    if (slice < M.nslices_split) cand_split_slice(M, S, slice);  // warp-uniform
    return;
  }
  const int slice = blockIdx.x;
  const int64_t c = (int64_t)slice * kSliceW + lane, vo = M.slice_off[slice] + lane;
  const SplitChunk x = split_chunk(M, S, c);  // the same in every warp
  if (__ballot_sync(kFull, x.rv.act != 0) == 0u) return;
  if (warp == 0)
    s_len[lane] =
        enqueue_named<kSliceW>(x.rv, x.t, x.mininf, x.maxinf, c, vo, S) ? x.len : 0;
  __syncthreads();
  const int32_t rlen = s_len[lane];
  if (__ballot_sync(kFull, rlen > 0) == 0u) return;
  enqueue_reread<kSliceW, false>(x.rv, rlen, warp * 4, kRoundWarps * 4, c, vo, M, M.col, S);
}

// ------------------------------------------------------------- k_finish --

constexpr int kFinishThreads = 256;

// Ends a round: the next state becomes the current one.  The last block to
// arrive (threadfence-reduction pattern; nobody waits) counts the round and
// sets the WHILE condition of the enclosing graph node.
// Commits one variable's next state (thread-level): the keys become the
// record the next round gathers; crossing bounds flag infeasibility.
template <bool kMulti>
__device__ __forceinline__ void finish_var(const DevState &S, const uint8_t *vartype, int64_t j,
                                           double eps_feas, float tau_dn, float eps_dn) {
  int32_t *inf_flag = &S.ctrl->infeasible;
  if (kMulti) {
    const int32_t inst = S.I.var_inst[j];
    if (S.I.done[inst]) return;  // a stopped problem keeps its bounds
    inf_flag = &S.I.infeasible[inst];
  }
  longlong2 kk = reinterpret_cast<const longlong2 *>(S.keys)[j];
  double L = val_of_key(kk.x), U = val_of_key(kk.y);
  uint32_t vt = vartype[j] ? 1u : 0u;
  if (kk.x > kk.y) {  // L > U in key order: test the crossing exactly
    bool cross = vt ? (L > U) : (L > U + eps_feas * d_max1abs(U));
    if (cross) set_flag(inf_flag);
  }
  write_var(S.rec + j, L, U, vt, tau_dn, eps_dn);
}

constexpr int kFinishWords = 8;  // bitmap words per warp and step of k_finish

// Commits the variables marked in words [w0, w0 + kFinishWords) of the
// dirty bitmap, clears those words and marks the variables' chunks for the
// next round if `mark` (warp-level, all 32 lanes): lanes read one word each,
// then the warp takes the changed variables 32 at a time.  kCo: masks are
// read through L2 (the persistent loop, where L1 may hold a word of an earlier
// round).  Returns the number of changed variables.  (Nothing here touches the
// control block: with a counter that every warp adds to, the commit of 1.5M
// variables took 140 us instead of 25, all of it waiting for that line.)
template <bool kMulti, bool kCo = false>
__device__ __forceinline__ int finish_words(const DevMatrix &M, const DevState &S,
                                            const uint8_t *vartype, int64_t w0, int64_t nwords,
                                            bool mark, double eps_feas, float tau_dn,
                                            float eps_dn) {
  const int lane = threadIdx.x & 31;
  const int64_t w = w0 + lane;
  uint32_t bits = 0u;
  if (lane < kFinishWords && w < nwords) {
    bits = S.dirty[w];
    if (bits) S.dirty[w] = 0u;
  }
  if (__ballot_sync(kFull, bits != 0u) == 0u) return 0;
  int incl = __popc(bits);  // over the lanes that hold words
#pragma unroll
  for (int o = 1; o < kFinishWords; o <<= 1) {
    const int v = __shfl_up_sync(kFull, incl, o);
    if (lane >= o) incl += v;
  }
  const int total = __shfl_sync(kFull, incl, kFinishWords - 1);
  for (int b0 = 0; b0 < total; b0 += 32) {
    const int k = b0 + lane;
    int src = 0;  // the word that holds the k-th changed variable
#pragma unroll
    for (int o = kFinishWords / 2; o > 0; o >>= 1) {
      const int v = __shfl_sync(kFull, incl, src + o - 1);
      if (v <= k) src += o;
    }
    const uint32_t wd = __shfl_sync(kFull, bits, src);
    const int below = __shfl_sync(kFull, incl, src) - __popc(wd);
    int32_t beg = 0, deg = 0;
    if (k < total) {
      const int64_t j = (w0 + src) * 32 + nth_bit(wd, k - below);
      if (mark) {
        beg = M.col_ptr[j];
        deg = M.col_ptr[j + 1] - beg;
      }
      finish_var<kMulti>(S, vartype, j, eps_feas, tau_dn, eps_dn);
    }
    if (!markable(deg)) {
      if (lane == 0) S.ctrl->all_next = 1;
    } else if (mark) {
      mark_columns<kCo>(M.col_slot, S.mask, beg, deg);
    }
  }
  return total;
}

// Ends a round (one block, all threads; after every variable is committed):
// counts the round, resets the round's counters and returns whether to
// continue.  For a problem set each problem counts its rounds and stops on
// its own (no change, infeasible, or the cap); the loop runs while any
// problem is live.
template <bool kMulti>
__device__ __forceinline__ int decide_round(const DevState &S) {
  volatile Ctrl *vc = S.ctrl;
  // every word before any decision, so that the loads overlap
  const int32_t r = vc->round + 1, max_rounds = vc->max_rounds, err = vc->err;
  const int32_t chg = vc->changed, infeasible = vc->infeasible, all_next = vc->all_next;
  const int32_t mark_now = vc->mark_now, mark_limit = vc->mark_limit, nch = vc->nchanged;
  int32_t cont;
  if (threadIdx.x < kQueues) S.qcount[threadIdx.x * kQueueStep] = 0;
  if (kMulti) {
    volatile int32_t *ch = S.I.changed, *inf = S.I.infeasible, *dn = S.I.done;
    int live = 0;
    for (int i = threadIdx.x; i < S.I.ninst; i += blockDim.x) {
      if (dn[i]) continue;
      const int32_t ri = S.I.rounds[i] + 1;
      S.I.rounds[i] = ri;
      int32_t d = 0;
      if (inf[i]) d = 1;
      else if (!ch[i]) d = 1;
      else if (ri >= max_rounds) {
        d = 1;
        S.I.status[i] = 1;
      }
      dn[i] = d;
      ch[i] = 0;
      live |= !d;
    }
    live = __syncthreads_or(live);
    cont = (live && !err && r < max_rounds) ? 1 : 0;
    if (threadIdx.x == 0) vc->last_changed = live;
  } else {
    cont = (chg && !infeasible && !err && r < max_rounds) ? 1 : 0;
    __syncthreads();
    if (threadIdx.x == 0) vc->last_changed = chg;
  }
  if (threadIdx.x == 0) {
    vc->round = r;
    vc->changed = 0;
    // The next round processes every chunk unless this one marked.  The next
    // round marks if it is expected to change few enough variables (rounds
    // change about three quarters of what the round before did).
    const bool all = all_next || !mark_now;
    vc->all_active = all;
    vc->sparse = !all && nch <= mark_limit / 32;
    vc->all_next = 0;
    vc->nchanged = 0;
    vc->mark_now = nch - nch / 4 <= mark_limit;
    vc->cont = cont;
    __threadfence();
  }
  return cont;
}

// Ends a round: every variable's next state becomes the current one.  The
// last block to arrive (threadfence-reduction pattern; nobody waits) decides
// whether to loop and sets the WHILE condition of the enclosing graph node.
template <bool kMulti>
__global__ void __launch_bounds__(kFinishThreads)
k_finish(DevMatrix M, DevState S, const uint8_t *vartype, cudaGraphConditionalHandle handle,
         int use_cond) {
  Ctrl *ctrl = S.ctrl;
  const int32_t err = ctrl->err;
  const double eps_feas = ctrl->eps_feas;
  const float tau_dn = f32_dn(ctrl->tau_rel), eps_dn = f32_dn(ctrl->eps_int);
  __shared__ int s_changed;
  if (threadIdx.x == 0) s_changed = 0;
  __syncthreads();
  if (!err) {  // only variables whose next state changed (the dirty bitmap)
    const bool mark = ctrl->mark_now != 0;
    int changed = 0;
    const int64_t nwords = ((int64_t)M.n + 31) >> 5;
    const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t w0 = warp * kFinishWords; w0 < nwords; w0 += nwarps * kFinishWords)
      changed += finish_words<kMulti>(M, S, vartype, w0, nwords, mark, eps_feas, tau_dn, eps_dn);
    if ((threadIdx.x & 31) == 0 && changed) atomicAdd(&s_changed, changed);
  }
  __shared__ int s_last;
  __syncthreads();
  if (threadIdx.x == 0) {
    if (s_changed) atomicAdd(&ctrl->nchanged, s_changed);
    __threadfence();
    unsigned prev = atomicAdd(&ctrl->blocks_done, 1u);
    s_last = prev == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  const int cont = decide_round<kMulti>(S);
  if (threadIdx.x == 0) {
    ctrl->blocks_done = 0;
    __threadfence();
    if (use_cond) cudaGraphSetConditional(handle, (unsigned)cont);
  }
}

// ------------------------------------------------------- persistent loop --
//
// The whole round loop as one cooperative launch (every block resident):
// the round's phases are separated by grid barriers instead of kernel
// boundaries, and the loop condition is read by every block after the last
// barrier of a round -- the paper's device-driven loop (Sec. 3.7) as a
// single persistent kernel, measured against the graph's WHILE node.

constexpr int kPersistThreads = 256;
// Grid-wide barrier (sense by generation count).  Bounded: a block that
// waits more than `limit` sleeps of 64 ns records DP_ERR_TIMEOUT and leaves;
// every block returns false once an error is recorded.  Cannot deadlock
// under a cooperative launch, which guarantees that all blocks are resident.
__device__ __forceinline__ bool grid_sync(const DevState &S, long long limit) {
  __syncthreads();
  if (threadIdx.x == 0) {
    volatile unsigned *gen = S.bar + 1;
    const unsigned g = *gen;
    __threadfence();
    if (atomicAdd(S.bar, 1u) == gridDim.x - 1) {
      S.bar[0] = 0u;  // every block has arrived; none leaves before gen moves
      __threadfence();
      atomicAdd(S.bar + 1, 1u);
    } else {
      long long it = 0;
      while (*gen == g) {
        if (++it > limit) {
          atomicExch(&S.ctrl->err, DP_ERR_TIMEOUT);
          break;
        }
        __nanosleep(64);
      }
    }
    __threadfence();
  }
  __syncthreads();
  return ((volatile Ctrl *)S.ctrl)->err == 0;
}

// Two resident blocks per SM: the union of all phases needs more registers
// than three blocks allow (spills), and fewer resident warps hide less latency.
// kMulti: a problem set (per-problem termination, as the graph's kernels).
template <bool kMulti>
__global__ void __launch_bounds__(kPersistThreads, 2)
k_persistent(DevMatrix M, DevState S, const uint8_t *vartype) {
  if (((volatile Ctrl *)S.ctrl)->err) return;  // set before the launch: uniform
  const Ctrl prm = *S.ctrl;  // parameters (constant during the run)
  const long long lim = prm.wait_limit;
  const float tau_dn = f32_dn(prm.tau_rel), eps_dn = f32_dn(prm.eps_int);
  const int wpb = kPersistThreads / 32;
  const int gw = blockIdx.x * wpb + (threadIdx.x >> 5), nw = gridDim.x * wpb;
  const int64_t gt = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t nt = (int64_t)gridDim.x * blockDim.x;
  for (;;) {
    const bool all = ((volatile Ctrl *)S.ctrl)->all_active != 0;
    for (int sl = gw; sl < M.nslices; sl += nw) {
      const uint32_t bits = take_mask(S, sl, all);
      if (bits == 0u) continue;
      if (M.val8) round_slice<kMulti, true, true>(M, S, sl, bits);
      else round_slice<kMulti, false, true>(M, S, sl, bits);
    }
    if (!grid_sync(S, lim)) return;
    if (M.nsplit_rows > 0) {
      for (int w = gw; w < M.nsplit_rows; w += nw) combine_rows<kMulti>(M, S, w);
      if (!grid_sync(S, lim)) return;
      for (int sl = gw; sl < M.nslices_split; sl += nw) cand_split_slice<true>(M, S, sl);
      if (!grid_sync(S, lim)) return;
    }
    if (cand_queues<kMulti, true>(M, S, prm) && !kMulti) S.ctrl->changed = 1;
    if (!grid_sync(S, lim)) return;
    const bool mark = ((volatile Ctrl *)S.ctrl)->mark_now != 0;
    const int64_t nwords = ((int64_t)M.n + 31) >> 5;
    int changed = 0;
    for (int64_t w0 = (gt >> 5) * kFinishWords; w0 < nwords; w0 += (nt >> 5) * kFinishWords)
      changed += finish_words<kMulti, true>(M, S, vartype, w0, nwords, mark, prm.eps_feas, tau_dn,
                                            eps_dn);
    if ((threadIdx.x & 31) == 0 && changed) atomicAdd(&S.ctrl->nchanged, changed);
    if (!grid_sync(S, lim)) return;
    if (blockIdx.x == 0) decide_round<kMulti>(S);
    if (!grid_sync(S, lim)) return;
    if (!((volatile Ctrl *)S.ctrl)->cont) return;
  }
}

// ------------------------------------------------------ prologue/epilogue --

// Normalises one call's inputs into the workspace: |v| >= inf_threshold
// becomes +-inf; integer bounds are rounded (ceil(lb - eps_int),
// floor(ub + eps_int)); NaN and contradictory infinities set ctrl->err.
__global__ void k_prologue(DevState S, uint8_t *vt_ws, int32_t m, int32_t n,
                           const double *lb, const double *ub, const uint8_t *vartype,
                           const double *lhs, const double *rhs, double eps_int,
                           double tau_rel, double thr) {
  const float tau_dn = f32_dn(tau_rel), eps_dn = f32_dn(eps_int);
  const double pinf = __longlong_as_double(0x7FF0000000000000ll);
  int64_t total = (int64_t)(n > m ? n : m);
  const int lane = threadIdx.x & 31;
  // warp-uniform loop (the block size and the stride are multiples of 32)
  for (int64_t i0 = blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31); i0 < total;
       i0 += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = i0 + lane;
    bool cross = false;
    if (i < n) {
      double L = lb[i], U = ub[i];
      uint8_t vt = vartype[i] ? 1 : 0;
      bool bad = d_isnan(L) || d_isnan(U) || L >= thr || U <= -thr;
      if (bad) {
        atomicExch(&S.ctrl->err, DP_ERR_NAN_INPUT);
        L = 0.0;
        U = 0.0;
      }
      if (L <= -thr) L = -pinf;
      if (U >= thr) U = pinf;
      if (vt) {
        if (d_isfinite(L)) L = ceil(L - eps_int);
        if (d_isfinite(U)) U = floor(U + eps_int);
      }
      reinterpret_cast<longlong2 *>(S.keys)[i] = make_longlong2(key_of(L), key_of(U));
      write_var(S.rec + i, L, U, vt, tau_dn, eps_dn);
      vt_ws[i] = vt;
      cross = key_of(L) > key_of(U);
    }
    // A round commits only the variables marked in the dirty bitmap; bounds
    // that cross on input are marked for round 1, whose commit tests them.
    // Writing whole words also clears what an aborted call left behind.
    const unsigned cw = __ballot_sync(kFull, cross);
    if (i0 < n && lane == 0) S.dirty[i0 >> 5] = cw;
    if (i < m) {
      double l = lhs[i], r = rhs[i];
      bool bad = d_isnan(l) || d_isnan(r) || l >= thr || r <= -thr;
      if (bad) {
        atomicExch(&S.ctrl->err, DP_ERR_NAN_INPUT);
        l = 0.0;
        r = 0.0;
      }
      if (l <= -thr) l = -pinf;
      if (r >= thr) r = pinf;
      S.lhs[i] = l;
      S.rhs[i] = r;
    }
  }
}

// Copies the normalised sides of each chunk's row into slot order, so that
// the round kernel reads them coalesced.
__global__ void k_prologue_sides(DevMatrix M, DevState S, const double *lhs, const double *rhs,
                                 double thr) {
  const double pinf = __longlong_as_double(0x7FF0000000000000ll);
  const int64_t nslots = (int64_t)M.nslices * kSliceW;
  for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < nslots;
       c += (int64_t)gridDim.x * blockDim.x) {
    const int32_t row = M.chunk_row[c];
    double l = 0.0, r = 0.0;
    if (row >= 0) {
      l = lhs[row];
      r = rhs[row];
      if (l <= -thr) l = -pinf;
      if (r >= thr) r = pinf;
    }
    S.side[c] = make_double2(l, r);
  }
  if (blockIdx.x == 0 && threadIdx.x < kQueues) S.qcount[threadIdx.x * kQueueStep] = 0;
  if (M.col_ptr == nullptr) return;
  // nothing is marked (the first round processes every chunk); an aborted
  // call may have left marks and touched rows behind
  for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
       c < M.nslices || c < M.nsplit_rows; c += (int64_t)gridDim.x * blockDim.x) {
    if (c < M.nslices) S.mask[c] = 0u;
    if (c < M.nsplit_rows) S.touch[c] = 0;
  }
}

__global__ void k_epilogue(DevState S, int32_t n, double *lb_out, double *ub_out) {
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < n;
       j += (int64_t)gridDim.x * blockDim.x) {
    longlong2 kk = reinterpret_cast<const longlong2 *>(S.keys)[j];
    lb_out[j] = val_of_key(kk.x);
    ub_out[j] = val_of_key(kk.y);
  }
}

// ------------------------------------------------------------ launchers --

static int grid_for(int64_t work, int threads, int max_blocks) {
  int64_t b = (work + threads - 1) / threads;
  if (b < 1) b = 1;
  if (b > max_blocks) b = max_blocks;
  return (int)b;
}

cudaError_t launch_prologue(const DevMatrix &M, const DevState &S, uint8_t *vt_ws, int32_t m,
                            int32_t n, const double *lb, const double *ub,
                            const uint8_t *vartype, const double *lhs, const double *rhs,
                            double eps_int, double tau_rel, double thr, int num_sms,
                            cudaStream_t st) {
  int64_t total = n > m ? n : m;
  k_prologue<<<grid_for(total, 256, num_sms * 16), 256, 0, st>>>(
      S, vt_ws, m, n, lb, ub, vartype, lhs, rhs, eps_int, tau_rel, thr);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (m > 0) {
    k_prologue_sides<<<grid_for((int64_t)M.nslices * kSliceW, 256, num_sms * 16), 256, 0, st>>>(
        M, S, lhs, rhs, thr);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess && M.layout == kLayoutMerge) e = launch_merge_prologue(M, S, st);
  return e;
}

cudaError_t launch_epilogue(const DevState &S, int32_t n, double *lb_out, double *ub_out,
                            int num_sms, cudaStream_t st) {
  k_epilogue<<<grid_for(n, 256, num_sms * 16), 256, 0, st>>>(S, n, lb_out, ub_out);
  return cudaGetLastError();
}

// The sliced-ELL part of a round: activities, split rows, Step 2 and the
// screen (events ev[0..5] as in launch_round_kernels).
template <bool kMulti, int kRoundWarps>
cudaError_t launch_ell_front(const DevMatrix &M, const DevState &S, int num_sms,
                             cudaStream_t st, cudaEvent_t *ev) {
  cudaError_t e;
  const int few = M.nlong <= kTeamBlocksPerSM * num_sms;
  int nb = M.nlong + (M.nslices - M.nlong + kRoundWarps - 1) / kRoundWarps;
  if (nb < 1) nb = 1;
  if (ev) cudaEventRecord(ev[0], st);
  if (M.val8)
    k_round<kMulti, kRoundWarps, true><<<nb, kRoundWarps * 32, 0, st>>>(M, S, few);
  else
    k_round<kMulti, kRoundWarps, false><<<nb, kRoundWarps * 32, 0, st>>>(M, S, few);
  if (ev) cudaEventRecord(ev[1], st);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if (M.nsplit_rows > 0) {
    int nbc = (M.nsplit_rows + kCombineWarps - 1) / kCombineWarps;  // a warp per row
    if (ev) cudaEventRecord(ev[2], st);
    k_combine<kMulti><<<nbc, kCombineWarps * 32, 0, st>>>(M, S);
    if (ev) cudaEventRecord(ev[3], st);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const int nbs = M.long_split + (M.nslices_split - M.long_split + kRoundWarps - 1) / kRoundWarps;
    if (ev) cudaEventRecord(ev[4], st);
    k_cand_split<kRoundWarps><<<nbs, kRoundWarps * 32, 0, st>>>(M, S);
    if (ev) cudaEventRecord(ev[5], st);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template <bool kMulti, int kRoundWarps>
cudaError_t launch_round_t(const DevMatrix &M, const DevState &S, const uint8_t *vt_ws,
                           cudaGraphConditionalHandle handle, int use_cond, int num_sms,
                           cudaStream_t st, cudaEvent_t *ev) {
  cudaError_t e = M.layout == kLayoutMerge ? launch_merge_front(M, S, num_sms, st, ev)
                                           : launch_ell_front<kMulti, kRoundWarps>(M, S, num_sms, st, ev);
  if (e != cudaSuccess) return e;
  // the queue kernel's grid: the blocks that are resident at once (a
  // larger grid-stride grid would run its last blocks as a second wave)
  static int queue_blocks_per_sm = 0;
  if (queue_blocks_per_sm == 0) {
    int b = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_cand_queue<kMulti>, 256, 0) !=
            cudaSuccess ||
        b < 1)
      b = 4;
    queue_blocks_per_sm = b;
  }
  if (ev) cudaEventRecord(ev[8], st);
  k_cand_queue<kMulti><<<num_sms * queue_blocks_per_sm, 256, 0, st>>>(M, S);
  if (ev) cudaEventRecord(ev[9], st);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  // one warp per kFinishWords bitmap words
  int nbf = grid_for(((int64_t)M.n + 31) / 32 * 32 / kFinishWords, kFinishThreads, num_sms * 6);
  if (ev) cudaEventRecord(ev[6], st);
  k_finish<kMulti><<<nbf, kFinishThreads, 0, st>>>(M, S, vt_ws, handle, use_cond);
  if (ev) cudaEventRecord(ev[7], st);
  return cudaGetLastError();
}

// Launches one round's kernels on `st`.  In the graph body (use_cond = 1)
// k_finish sets the WHILE condition; in the host-driven loop it does not.
// With `ev` (10 events) each kernel is bracketed by a pair of events.  A
// problem set (S.I.ninst > 0) runs the per-problem variants.
cudaError_t launch_round_kernels(const DevMatrix &M, const DevState &S, const uint8_t *vt_ws,
                                 cudaGraphConditionalHandle handle, int use_cond, int num_sms,
                                 cudaStream_t st, cudaEvent_t *ev) {
  const bool w4 = M.round_warps == 4;
  if (S.I.ninst > 0)
    return w4 ? launch_round_t<true, 4>(M, S, vt_ws, handle, use_cond, num_sms, st, ev)
              : launch_round_t<true, 8>(M, S, vt_ws, handle, use_cond, num_sms, st, ev);
  return w4 ? launch_round_t<false, 4>(M, S, vt_ws, handle, use_cond, num_sms, st, ev)
            : launch_round_t<false, 8>(M, S, vt_ws, handle, use_cond, num_sms, st, ev);
}

cudaError_t launch_persistent(const DevMatrix &M, const DevState &S, const uint8_t *vt_ws,
                              int num_sms, cudaStream_t st) {
  const void *kern = S.I.ninst > 0 ? (const void *)k_persistent<true>
                                    : (const void *)k_persistent<false>;
  int per_sm = 0;
  cudaError_t e =
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kPersistThreads, 0);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorLaunchOutOfResources;
  if ((e = cudaMemsetAsync(S.bar, 0, 2 * sizeof(unsigned), st)) != cudaSuccess) return e;
  DevMatrix m = M;
  DevState s = S;
  const uint8_t *vt = vt_ws;
  void *args[] = {&m, &s, &vt};
  return cudaLaunchCooperativeKernel(kern, dim3(num_sms * per_sm), dim3(kPersistThreads), args,
                                     0, st);
}

cudaError_t launch_round_body(const DevMatrix &M, const DevState &S, const uint8_t *vt_ws,
                              cudaGraphConditionalHandle handle, int num_sms,
                              cudaStream_t st) {
  return launch_round_kernels(M, S, vt_ws, handle, 1, num_sms, st, nullptr);
}

}  // namespace dp
