// Round helpers shared by the sliced-ELL kernels (dp_kernels.cu) and the
// merge-path kernels (dp_merge.cu): the per-side top-2 of the binary32
// screen values and the queueing of the nonzeros that survive the screen.
#pragma once
#include "dp_device.cuh"

namespace dp {

__device__ __forceinline__ void top2_add(float t, int k, float &t1, float &t2, int32_t &k1) {
  if (t > t1) {
    t2 = t1;
    t1 = t;
    k1 = k;
  } else if (t > t2) {
    t2 = t;
  }
}

// Adds another part's top-2 (s1 >= s2, slot ks of s1).
__device__ __forceinline__ void top2_merge(float s1, float s2, int ks, float &t1, float &t2,
                                           int32_t &k1) {
  if (s1 > t1) {
    t2 = fmaxf(t1, s2);
    t1 = s1;
    k1 = ks;
  } else {
    t2 = fmaxf(t2, s1);
  }
}

__device__ __forceinline__ Top2 top2_init() {
  Top2 t;
  t.r1 = t.r2 = t.l1 = t.l2 = -f_inf();
  t.kr = t.kl = 0;
  t.kinf_min = t.kinf_max = 0;
  return t;
}

// ---- rows of at most kMax nonzeros ----
//
// A lane keeps the screen values of such a row in registers (the loops over
// its slots are unrolled), so that the survivors are known from the row's
// thresholds without another pass over its nonzeros, and the running top-2 of
// the longer rows is not needed either.
// What the unrolled pass leaves: kSides = 1: one side's sums and values,
// kSides = 2: the minimum activity first, then the maximum.
template <int kSides, int kMax>
struct ShortAct {
  double fin[kSides];
  int32_t ninf[kSides], kinf[kSides];
  float t[kSides][kMax];
};

// Activity sums, infinity counts and screen values of the lane's row (len <=
// kMax slots from elem0, stride kSliceW; 0 for none).  kSides = 1:
// `right` selects the minimum activity (the right-hand side's), else the
// maximum.  rec(j, L, U, WU, WL) loads a record.  The sums are one FMA chain
// in CSR order.  All 32 lanes call.
template <int kSides, int kMax, class Rec>
__device__ __forceinline__ void short_activity(const DevMatrix &M, int64_t elem0, int32_t len,
                                               bool right, Rec rec,
                                               ShortAct<kSides, kMax> &r) {
  constexpr int kG = 4;
  const int maxlen = __reduce_max_sync(kFull, len);
  const double *vp = M.val + elem0;
  const int32_t *cp = M.col + elem0;
#pragma unroll
  for (int s = 0; s < kSides; ++s) {
    r.fin[s] = 0.0;
    r.ninf[s] = r.kinf[s] = 0;
  }
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
#pragma unroll
  for (int g = 0; g < kMax / kG; ++g) {
    if (g > 0 && g * kG >= maxlen) {  // warp-uniform
#pragma unroll
      for (int u = 0; u < kG; ++u)
#pragma unroll
        for (int s = 0; s < kSides; ++s) r.t[s][g * kG + u] = -f_inf();
      continue;
    }
    double a[kG], L[kG], U[kG];
    float WU[kG], WL[kG];
#pragma unroll
    for (int u = 0; u < kG; ++u) {
      a[u] = an[u];
      L[u] = U[u] = 0.0;
      WU[u] = WL[u] = 0.0f;
      if (g * kG + u < len) rec(jn[u], L[u], U[u], WU[u], WL[u]);
    }
    if ((g + 1) * kG < kMax && (g + 1) * kG < maxlen) {
#pragma unroll
      for (int u = 0; u < kG; ++u) {
        an[u] = 1.0;
        jn[u] = 0;
        if ((g + 1) * kG + u < len) {
          an[u] = __ldcs(vp + ((g + 1) * kG + u) * kSliceW);
          jn[u] = __ldcs(cp + ((g + 1) * kG + u) * kSliceW);
        }
      }
    }
#pragma unroll
    for (int u = 0; u < kG; ++u) {
      const int k = g * kG + u;
      const float au = absup_fast(a[u]), ad = absdn_fast(a[u]);
#pragma unroll
      for (int s = 0; s < kSides; ++s) {
        const bool low = d_pos(a[u]) == (kSides == 2 ? s == 0 : right);
        const double b = low ? L[u] : U[u];
        const bool inf = d_isinf(b);
        const float t = screen_prod(au, ad, low ? WU[u] : WL[u]);
        r.t[s][k] = k < len ? t : -f_inf();
        if (k < len) {
          r.ninf[s] += inf;
          if (inf) r.kinf[s] = k;
          r.fin[s] = fma(a[u], inf ? 0.0 : b, r.fin[s]);
        }
      }
    }
  }
}

// The largest screen value of a side.
template <int kMax>
__device__ __forceinline__ float short_max(const float (&t)[kMax]) {
  float m = t[0];
#pragma unroll
  for (int k = 1; k < kMax; ++k) m = fmaxf(m, t[k]);
  return m;
}

// The slots of a row that survive one side's screen (bit k: slot k); `fin`:
// the side is finite.
template <int kMax>
__device__ __forceinline__ uint32_t short_survivors(const float (&t)[kMax], int32_t len,
                                                    bool fin, int32_t ninf, int32_t kinf,
                                                    float thr, bool exact) {
  if (!fin || ninf > 1) return 0u;
  if (ninf == 1) return 1u << kinf;
  const uint32_t all = (1u << len) - 1u;
  if (exact) return f_inf() > thr ? all : 0u;
  uint32_t m = 0u;
#pragma unroll
  for (int k = 0; k < kMax; ++k)
    if (t[k] > thr) m |= 1u << k;
  return m & all;
}

// Reserves c (0..15) consecutive entries per lane in the queue of chunk slots
// slot..slot+31 with one atomic per warp (all 32 lanes call): the lanes'
// offsets come from ballots of the bits of c (kBits of them), not from a
// shuffle scan.  Returns the lane's first entry
// (meaningless when c = 0).
template <int kBits = 3>
__device__ __forceinline__ uint32_t warp_reserve(int c, int64_t slot, const DevState &S) {
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  int total = 0, before = 0;
#pragma unroll
  for (int k = 0; k < kBits; ++k) {
    const unsigned b = __ballot_sync(kFull, c & (1 << k));
    total += __popc(b) << k;
    before += __popc(b & lt) << k;
  }
  if (total == 0) return 0u;
  uint32_t base = 0u;
  if (lane == 0) {
    const int q = (int)(slot >> 5) % kQueues;
    base = S.qbase[q] + (uint32_t)atomicAdd(S.qcount + q * kQueueStep, total);
  }
  return __shfl_sync(kFull, base, 0) + (uint32_t)before;
}

// Queueing of the nonzeros of the lanes' chunks whose candidates survive
// the screen.  Entries go to a global queue (warp-aggregated slots) and are
// evaluated by k_cand_queue, one per thread, so the binary64 candidate
// formulas run lane-dense across the whole GPU however few survivors a warp
// has.  When the second-largest screen value of a side is below the
// threshold, only the chunk's largest can survive and it is queued directly
// (enqueue_named, no re-read); otherwise the chunk is re-read
// (enqueue_reread: values and columns from L2, records through the same
// gather), four slots at a time.  Element k of a lane's chunk sits at
// elem0 + k * kStride of val/col (slot-major slices: the lane's slot in the
// slice, stride 32; CSR rows: the row's offset, stride 1).

__device__ __forceinline__ CandEntry cand_entry(int64_t elem, int64_t chunk_slot,
                                                unsigned sides) {
  CandEntry e;
  e.off = (uint32_t)elem;
  e.cs = ((uint32_t)chunk_slot << 2) | sides;
  return e;
}

__device__ __forceinline__ void put_rowsum(const RowView &mine, int64_t chunk_slot,
                                           const DevState &S) {
  RowSum rs;
  rs.minfin = mine.minfin;
  rs.maxfin = mine.maxfin;
  rs.mininf = mine.mininf;
  rs.maxinf = mine.maxinf;
  S.rowsum[chunk_slot] = rs;
}

// Queues the survivors that can be named without re-reading the chunk and
// writes the row's sums for every lane that has, or may have, an entry.
// Returns whether the lane's chunk needs the re-read.  All 32 lanes call.
template <int kStride>
__device__ __forceinline__ bool enqueue_named(const RowView &mine, const Top2 &t,
                                              int chunk_mininf, int chunk_maxinf,
                                              int64_t chunk_slot, int64_t elem0,
                                              const DevState &S) {
  const bool act = mine.act != 0;
  if (__ballot_sync(kFull, act) == 0u) return false;
  // Survivors can be named unless a side has two screen values above its
  // threshold (or the row skips the screen).  With exactly one infinite
  // contribution to a side's activity, only that nonzero gets a finite
  // residual on that side (Sec. 3.4); its slot was recorded by the activity
  // pass.
  const bool full = act && (mine.exact || (mine.mininf == 0 && t.r2 > mine.thr_r) ||
                            (mine.maxinf == 0 && t.l2 > mine.thr_l));
  bool h1 = false, h2 = false;
  int k1 = 0, k2 = 0;
  if (act && !full) {
    const bool fr = d_isfinite(mine.rhs), fl = d_isfinite(mine.lhs);
    if (fr && mine.mininf == 0 && t.r1 > mine.thr_r) { h1 = true; k1 = t.kr; }
    if (fr && mine.mininf == 1 && chunk_mininf > 0) { h1 = true; k1 = t.kinf_min; }
    if (fl && mine.maxinf == 0 && t.l1 > mine.thr_l) { h2 = true; k2 = t.kl; }
    if (fl && mine.maxinf == 1 && chunk_maxinf > 0) { h2 = true; k2 = t.kinf_max; }
  }
  const bool merge = h1 && h2 && k1 == k2;
  const bool q2 = h2 && !merge;
  uint32_t pos = warp_reserve((h1 ? 1 : 0) + (q2 ? 1 : 0), chunk_slot, S);
  if (h1 || q2 || full) put_rowsum(mine, chunk_slot, S);
  if (h1) S.queue[pos++] = cand_entry(elem0 + (int64_t)k1 * kStride, chunk_slot, merge ? 3u : 1u);
  if (q2) S.queue[pos] = cand_entry(elem0 + (int64_t)k2 * kStride, chunk_slot, 2u);
  return full;
}

// Re-reads the lanes' chunks (len slots each, 0 for a lane without one) and
// queues every nonzero that survives the screen: four slots from `kbeg`,
// then every `kstep` slots further on (several warps can share the slots of
// a slice).  kCo: records are loaded through L2 (the persistent loop, which
// rewrites them between its phases).  All 32 lanes call.
template <int kStride, bool kCo>
__device__ __forceinline__ void enqueue_reread(const RowView &mine, int32_t len, int kbeg,
                                               int kstep, int64_t chunk_slot, int64_t elem0,
                                               const DevMatrix &M, const int32_t *col,
                                               const DevState &S) {
  const int maxlen = __reduce_max_sync(kFull, len);
  const int32_t *cp = col + elem0;
  // software-pipelined: the next group's values and columns are fetched
  // while this group's records are gathered
  double an[4];
  int32_t jn[4];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      an[u] = 1.0;
      jn[u] = 0;
      if (k0 + u < len) {
        an[u] = ld_coef(M, elem0 + (int64_t)(k0 + u) * kStride);
        jn[u] = cp[(int64_t)(k0 + u) * kStride];
      }
    }
  };
  if (kbeg < maxlen) fetch(kbeg);
  for (int k = kbeg; k < maxlen; k += kstep) {
    double a[4], L[4], U[4];
    float WU[4], WL[4];
    uint32_t fl[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      a[u] = an[u];
      L[u] = U[u] = 0.0;
      WU[u] = WL[u] = 0.0f;
      if (k + u < len) ld_rec_t<kCo>(S.rec + jn[u], L[u], U[u], WU[u], WL[u], fl[u]);
    }
    if (k + kstep < maxlen) fetch(k + kstep);
    unsigned sd[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      sd[u] = k + u < len ? nnz_sides(a[u], L[u], U[u], WU[u], WL[u], mine) : 0u;
    // one reservation for the group's survivors of all lanes
    int c = 0;
#pragma unroll
    for (int u = 0; u < 4; ++u) c += sd[u] != 0u;
    uint32_t pos = warp_reserve(c, chunk_slot, S);
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (sd[u] != 0u)
        S.queue[pos++] = cand_entry(elem0 + (int64_t)(k + u) * kStride, chunk_slot, sd[u]);
  }
}

// Both, by one warp.  Returns whether the lane's chunk needed the re-read
// (done here for its first mylen slots).
template <int kStride, bool kCo = false>
__device__ __forceinline__ bool warp_enqueue(const RowView &mine, const Top2 &t, int chunk_mininf,
                                             int chunk_maxinf, int32_t mylen, int64_t chunk_slot,
                                             int64_t elem0, const DevMatrix &M,
                                             const int32_t *col, const DevState &S) {
  const bool full =
      enqueue_named<kStride>(mine, t, chunk_mininf, chunk_maxinf, chunk_slot, elem0, S);
  if (__ballot_sync(kFull, full) == 0u) return false;
  enqueue_reread<kStride, kCo>(mine, full ? mylen : 0, 0, 4, chunk_slot, elem0, M, col, S);
  return full;
}

// ---- marking ----

// Position of the k-th set bit (k from 0) of a word that has more than k.
__device__ __forceinline__ int nth_bit(uint32_t w, int k) {
  int at = 0;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const int c = __popc((w >> at) & ((1u << o) - 1u));
    if (k >= c) {
      k -= c;
      at += o;
    }
  }
  return at;
}

// Whether the lists of the lanes' variables (deg entries each) are short enough
// for the warp to walk; if not, the next round processes every chunk.  A walk
// takes 0.25 us per 128 entries: without a limit the columns of a system with
// few variables took longer than the rounds they saved (48 variables, 90k
// nonzeros: 134 us per round, 20 with every chunk processed; a limit of 2048
// entries leaves 500 variables at 510 us per call where 512 gives 385).
// All 32 lanes call.
constexpr int32_t kMarkEntries = 512;
__device__ __forceinline__ bool markable(int32_t deg) {
  return __reduce_add_sync(kFull, min(deg, kMarkEntries + 1)) <= kMarkEntries;
}

// Marks the chunks of the lanes' variables (deg list entries each from beg;
// deg = 0 for none): the lists are walked as one sequence, so that the lanes
// stay busy whatever the column lengths.  A mask only gains bits while a
// round is committed, so a word that is seen, possibly in an older state, to
// have the bit needs no atomic.  kCo: the masks are read through L2 (needed
// where L1 may hold a word of an earlier round).  All 32 lanes call.
template <bool kCo>
__device__ __forceinline__ void mark_columns(const int32_t *col_slot, uint32_t *mask, int32_t beg,
                                             int32_t deg) {
  const int lane = threadIdx.x & 31;
  int32_t incl = deg;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int32_t v = __shfl_up_sync(kFull, incl, o);
    if (lane >= o) incl += v;
  }
  const int32_t total = __shfl_sync(kFull, incl, 31);
  const int32_t shift = beg - (incl - deg);  // list offset of sequence position 0
  for (int32_t e0 = 0; e0 < total; e0 += 128) {
    int32_t slot[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int32_t e = e0 + 32 * u + lane;
      int src = 0;  // the variable whose list holds position e
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const int32_t v = __shfl_sync(kFull, incl, src + o - 1);
        if (v <= e) src += o;
      }
      const int32_t sh = __shfl_sync(kFull, shift, src & 31);
      slot[u] = e < total ? __ldg(col_slot + e + sh) : -1;
    }
    uint32_t w[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const uint32_t *q = mask + (slot[u] >> 5);
      w[u] = slot[u] < 0 ? 0u : (kCo ? __ldcg(q) : __ldca(q));
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const uint32_t bit = 1u << (slot[u] & 31);
      if (slot[u] >= 0 && !(w[u] & bit)) atomicOr(mask + (slot[u] >> 5), bit);
    }
  }
}

// Appends one queue entry per lane with h set (warp-aggregated; all 32
// lanes call): element offset `off` of a row whose sums are at rowsum[slot].
__device__ __forceinline__ void warp_push(bool h, int64_t off, int64_t slot, unsigned sides,
                                          const DevState &S) {
  const unsigned pm = __ballot_sync(kFull, h);
  if (pm == 0u) return;
  const int lane = threadIdx.x & 31;
  const int leader = __ffs(pm) - 1;
  uint32_t base = 0u;
  if (lane == leader) {
    const int q = (int)(slot >> 5) % kQueues;
    base = S.qbase[q] + (uint32_t)atomicAdd(S.qcount + q * kQueueStep, __popc(pm));
  }
  base = __shfl_sync(kFull, base, leader);
  if (!h) return;
  CandEntry e;
  e.off = (uint32_t)off;
  e.cs = ((uint32_t)slot << 2) | sides;
  S.queue[base + __popc(pm & ((1u << lane) - 1u))] = e;
}

}  // namespace dp
