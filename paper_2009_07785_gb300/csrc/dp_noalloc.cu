// Allocation-free propagation entry point (dp_propagate_noalloc).
//
// Who needs it: callers that must not call cudaMalloc/cudaFree themselves or
// through a library -- for example a solver embedded in a process whose
// device memory belongs to a pool allocator (PyTorch's caching allocator, a
// MIP solver's own arena), where a stray cudaMalloc fragments or exhausts the
// pool, or a latency-sensitive pipeline where cudaMalloc/cudaFree would
// synchronise the device.  dp_matrix_load allocates the matrix's device
// layout and workspace; this entry point instead works directly on a CSR
// matrix and problem the caller already holds in device memory, and keeps
// its only scratch (the next-state bound keys and a control block) in one
// file-scope __device__ array of fixed size.
//
// The scratch array is shared by every call in the process on a given
// device and keeps the previous call's contents; each call re-initialises
// what it uses.  Calls whose GPU work overlaps (two streams, two host
// threads) race on it and must be serialised by the caller.
#include <cuda_runtime.h>
#include <atomic>
#include <cstdint>
#include <cstring>

#include "../../include/domprop.h"
#include "dp_trace.h"

namespace {

// next-state keys (2 per variable) followed by the control block
constexpr size_t kNoallocCtrlWords = 32;  // int64 words reserved for the control block
constexpr size_t kNoallocWords = 2 * (size_t)DP_NOALLOC_MAX_VARS + kNoallocCtrlWords;

__device__ __align__(256) long long g_noalloc_scratch[kNoallocWords];

// control block layout inside the scratch array (int32 view)
struct NoallocCtrl {
  int32_t err, changed, infeasible, pad;
};

constexpr int kMaxDevices = 64;
// Device address of the array, per device.  Host threads that call the entry
// point on different devices may fill their entries concurrently; the lookup
// is idempotent, so an atomic store per entry is all the synchronisation it
// needs.
std::atomic<long long *> g_scratch_addr[kMaxDevices] = {};

__device__ __forceinline__ bool is_inf_d(double x) {
  return ((unsigned long long)__double_as_longlong(x) << 1) == 0xFFE0000000000000ull;
}
__device__ __forceinline__ bool is_finite_d(double x) {
  return ((__double2hiint(x) >> 20) & 0x7FF) != 0x7FF;
}
__device__ __forceinline__ bool is_nan_d(double x) {
  return ((unsigned long long)__double_as_longlong(x) << 1) > 0xFFE0000000000000ull;
}
__device__ __forceinline__ long long okey(double x) {
  long long b = __double_as_longlong(x);
  return b >= 0 ? b : (b ^ 0x7FFFFFFFFFFFFFFFll);
}
__device__ __forceinline__ double okey_val(long long k) {
  return __longlong_as_double(k >= 0 ? k : (k ^ 0x7FFFFFFFFFFFFFFFll));
}
__device__ __forceinline__ double side_norm(double v, double thr) {
  const double pinf = __longlong_as_double(0x7FF0000000000000ll);
  if (v >= thr) return pinf;
  if (v <= -thr) return -pinf;
  return v;
}

// Checks the caller's CSR (so that no later kernel can read out of range)
// and normalises the bounds into the outputs (the round state) and keys.
__global__ void k_na_prologue(int32_t m, int32_t n, const int64_t *row_ptr,
                              const int32_t *col, const double *val, int64_t nnz,
                              const double *lb, const double *ub, const uint8_t *vt,
                              const double *lhs, const double *rhs, double eps_int, double thr,
                              double *lo, double *hi, long long *keys, NoallocCtrl *ctrl) {
  const double pinf = __longlong_as_double(0x7FF0000000000000ll);
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nnz; i += stride) {
    double a = val[i];
    if (col[i] < 0 || col[i] >= n || !is_finite_d(a) || a == 0.0) atomicExch(&ctrl->err, DP_ERR_BAD_CSR);
  }
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i <= m; i += stride) {
    if (i == 0 && row_ptr[0] != 0) atomicExch(&ctrl->err, DP_ERR_BAD_CSR);
    if (i == m && row_ptr[m] != nnz) atomicExch(&ctrl->err, DP_ERR_BAD_CSR);
    if (i < m && row_ptr[i + 1] < row_ptr[i]) atomicExch(&ctrl->err, DP_ERR_BAD_CSR);
    if (i < m) {
      double l = lhs[i], r = rhs[i];
      if (is_nan_d(l) || is_nan_d(r) || l >= thr || r <= -thr) atomicExch(&ctrl->err, DP_ERR_NAN_INPUT);
    }
  }
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < n; j += stride) {
    double L = lb[j], U = ub[j];
    if (is_nan_d(L) || is_nan_d(U) || L >= thr || U <= -thr) {
      atomicExch(&ctrl->err, DP_ERR_NAN_INPUT);
      L = U = 0.0;
    }
    if (L <= -thr) L = -pinf;
    if (U >= thr) U = pinf;
    if (vt[j]) {
      if (is_finite_d(L)) L = ceil(L - eps_int);
      if (is_finite_d(U)) U = floor(U + eps_int);
    }
    lo[j] = L;
    hi[j] = U;
    keys[2 * j] = okey(L);
    keys[2 * j + 1] = okey(U);
  }
}

// A row's sums and sides.
struct NaRow {
  double minfin, maxfin, lhs, rhs;
  int mininf, maxinf;
};

struct NaArgs {
  const int32_t *col;
  const double *val;
  const uint8_t *vt;
  const double *lo, *hi;
  long long *keys;
  NoallocCtrl *ctrl;
  double eps_int, tau, eps_feas, thr;
};

// One nonzero's contribution to the infinity counts; bn, bx: the bounds of
// the finite sums (0 in the place of an infinite one).
__device__ __forceinline__ void na_count(double a, double L, double U, NaRow &r, double &bn,
                                         double &bx) {
  const bool pos = __double2hiint(a) >= 0;
  bn = pos ? L : U;
  bx = pos ? U : L;
  if (is_inf_d(bn)) {
    ++r.mininf;
    bn = 0.0;
  }
  if (is_inf_d(bx)) {
    ++r.maxinf;
    bx = 0.0;
  }
}

// Step 2 of a row.
__device__ __forceinline__ void na_step2(const NaArgs &A, const NaRow &r) {
  if (r.mininf == 0 && is_finite_d(r.rhs) &&
      r.minfin > r.rhs + A.eps_feas * fmax(1.0, fabs(r.rhs)))
    atomicExch(&A.ctrl->infeasible, 1);
  if (r.maxinf == 0 && is_finite_d(r.lhs) &&
      r.maxfin < r.lhs - A.eps_feas * fmax(1.0, fabs(r.lhs)))
    atomicExch(&A.ctrl->infeasible, 1);
}

// One nonzero's candidates (Eq. 3a/3b in residual form, Eq. 5a/5b, the
// exactly-one-infinity rule), integer rounding and filtered atomics into the
// next-state keys.
__device__ __forceinline__ void na_candidates(const NaArgs &A, const NaRow &r, double a,
                                              int32_t j, double L, double U) {
  const bool pos = __double2hiint(a) >= 0;
  const double bmin = pos ? L : U, bmax = pos ? U : L;
  const bool have_r = is_finite_d(r.rhs) &&
                      (r.mininf == 0 || (r.mininf == 1 && is_inf_d(bmin)));
  const bool have_l = is_finite_d(r.lhs) &&
                      (r.maxinf == 0 || (r.maxinf == 1 && is_inf_d(bmax)));
  if (!have_r && !have_l) return;
  bool hl = false, hu = false;
  double lc = 0.0, uc = 0.0;
  if (have_r) {
    const double res = r.mininf == 0 ? fma(-a, bmin, r.minfin) : r.minfin;
    if (is_finite_d(res)) {
      const double c = (r.rhs - res) / a;
      if (pos) { uc = c; hu = true; } else { lc = c; hl = true; }
    }
  }
  if (have_l) {
    const double res = r.maxinf == 0 ? fma(-a, bmax, r.maxfin) : r.maxfin;
    if (is_finite_d(res)) {
      const double c = (r.lhs - res) / a;
      if (pos) { lc = c; hl = true; } else { uc = c; hu = true; }
    }
  }
  const bool isint = A.vt[j] != 0;
  if (hl) {
    if (isint) lc = ceil(lc - A.eps_int);
    if (!(fabs(lc) < A.thr)) hl = false;
  }
  if (hu) {
    if (isint) uc = floor(uc + A.eps_int);
    if (!(fabs(uc) < A.thr)) hu = false;
  }
  if (hl) {
    const bool acc = is_inf_d(L) || (isint ? lc > L : lc > L + A.tau * fmax(1.0, fabs(L)));
    if (acc) {
      atomicMax(&A.keys[2 * (int64_t)j], okey(lc));
      A.ctrl->changed = 1;
    }
  }
  if (hu) {
    const bool acc = is_inf_d(U) || (isint ? uc < U : uc < U - A.tau * fmax(1.0, fabs(U)));
    if (acc) {
      atomicMin(&A.keys[2 * (int64_t)j + 1], okey(uc));
      A.ctrl->changed = 1;
    }
  }
}

constexpr int kNaThreads = 256;
constexpr int kNaWarps = kNaThreads / 32;
constexpr int kNaBlocksPerSM = 3;  // resident blocks of k_na_round
constexpr int kNaUnroll = 4;     // nonzeros whose loads are in flight together
constexpr int kNaLaneRow = 32;   // longest row that one lane takes
constexpr int kNaWarpRow = 256;  // longest row that one warp takes
// What a row costs, in 0.062 us: a lane 2.1 us per nonzero (its candidates'
// divisions, whatever the other lanes do), a warp 4 us and 0.06 (few accepted
// candidates) to 0.12 us per nonzero, a block 8 us and 0.012 us per nonzero.
constexpr unsigned kNaLaneCost = 34, kNaWarpCost = 64, kNaBlockCost = 130, kNaBlockShare = 5;

// Loads nonzeros k, k + step, ... (kNaUnroll of them, those below e).
__device__ __forceinline__ void na_load(const NaArgs &A, int64_t k, int64_t step, int64_t e,
                                        double (&a)[kNaUnroll], int32_t (&j)[kNaUnroll],
                                        double (&L)[kNaUnroll], double (&U)[kNaUnroll]) {
#pragma unroll
  for (int u = 0; u < kNaUnroll; ++u) {
    a[u] = 1.0;
    j[u] = 0;
    if (k + u * step < e) {
      a[u] = A.val[k + u * step];
      j[u] = A.col[k + u * step];
    }
  }
#pragma unroll
  for (int u = 0; u < kNaUnroll; ++u) {
    L[u] = U[u] = 0.0;
    if (k + u * step < e) {
      L[u] = A.lo[j[u]];
      U[u] = A.hi[j[u]];
    }
  }
}

// A row by one lane: the activity chain in CSR order, Step 2, candidates.
__device__ __forceinline__ void na_row_lane(const NaArgs &A, NaRow r, int64_t b, int64_t e) {
  double a[kNaUnroll], L[kNaUnroll], U[kNaUnroll];
  int32_t j[kNaUnroll];
  for (int64_t k = b; k < e; k += kNaUnroll) {
    na_load(A, k, 1, e, a, j, L, U);
#pragma unroll
    for (int u = 0; u < kNaUnroll; ++u)
      if (k + u < e) {
        double bn, bx;
        na_count(a[u], L[u], U[u], r, bn, bx);
        r.minfin = fma(a[u], bn, r.minfin);
        r.maxfin = fma(a[u], bx, r.maxfin);
      }
  }
  na_step2(A, r);
  if (r.mininf > 1 && r.maxinf > 1) return;
  for (int64_t k = b; k < e; k += kNaUnroll) {
    na_load(A, k, 1, e, a, j, L, U);
#pragma unroll
    for (int u = 0; u < kNaUnroll; ++u)
      if (k + u < e) na_candidates(A, r, a[u], j[u], L[u], U[u]);
  }
}

// A row by one warp: 32 nonzeros are loaded side by side and added in CSR
// order over shuffled values (lanes below 16 the minimum activity, the
// others the maximum): the same chain as one lane's, bit for bit.
__device__ __forceinline__ void na_row_warp(const NaArgs &A, NaRow r, int64_t b, int64_t e) {
  const unsigned full = 0xFFFFFFFFu;
  const int lane = threadIdx.x & 31;
  double a[kNaUnroll], L[kNaUnroll], U[kNaUnroll];
  int32_t j[kNaUnroll];
  double fin = 0.0;
  for (int64_t k = b; k < e; k += 32 * kNaUnroll) {
    na_load(A, k + lane, 32, e, a, j, L, U);
#pragma unroll
    for (int u = 0; u < kNaUnroll; ++u) {
      double bn = 0.0, bx = 0.0;
      const int64_t k0 = k + 32 * u;
      if (k0 + lane < e) na_count(a[u], L[u], U[u], r, bn, bx);
      const int cnt = (int)(e - k0 < 32 ? e - k0 : 32);
      for (int i = 0; i < cnt; ++i) {  // warp-uniform
        const double av = __shfl_sync(full, a[u], i);
        const double vn = __shfl_sync(full, bn, i), vx = __shfl_sync(full, bx, i);
        fin = fma(av, lane < 16 ? vn : vx, fin);
      }
    }
  }
  r.minfin = __shfl_sync(full, fin, 0);
  r.maxfin = __shfl_sync(full, fin, 16);
  r.mininf = __reduce_add_sync(full, r.mininf);
  r.maxinf = __reduce_add_sync(full, r.maxinf);
  if (lane == 0) na_step2(A, r);
  if (r.mininf > 1 && r.maxinf > 1) return;
  for (int64_t k = b; k < e; k += 32 * kNaUnroll) {
    na_load(A, k + lane, 32, e, a, j, L, U);
#pragma unroll
    for (int u = 0; u < kNaUnroll; ++u)
      if (k + 32 * u + lane < e) na_candidates(A, r, a[u], j[u], L[u], U[u]);
  }
}

// A row by the whole block: every thread adds its strided nonzeros in order,
// then the threads' sums are added in a fixed tree, the same for every run.
__device__ __forceinline__ void na_row_block(const NaArgs &A, NaRow r, int64_t b, int64_t e) {
  __shared__ double s_min[kNaWarps], s_max[kNaWarps];
  __shared__ int s_ni[kNaWarps], s_xi[kNaWarps];
  const unsigned full = 0xFFFFFFFFu;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double a[kNaUnroll], L[kNaUnroll], U[kNaUnroll];
  int32_t j[kNaUnroll];
  for (int64_t k = b + threadIdx.x; k < e; k += kNaThreads * kNaUnroll) {
    na_load(A, k, kNaThreads, e, a, j, L, U);
#pragma unroll
    for (int u = 0; u < kNaUnroll; ++u)
      if (k + u * kNaThreads < e) {
        double bn, bx;
        na_count(a[u], L[u], U[u], r, bn, bx);
        r.minfin = fma(a[u], bn, r.minfin);
        r.maxfin = fma(a[u], bx, r.maxfin);
      }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    r.minfin += __shfl_xor_sync(full, r.minfin, o);
    r.maxfin += __shfl_xor_sync(full, r.maxfin, o);
  }
  r.mininf = __reduce_add_sync(full, r.mininf);
  r.maxinf = __reduce_add_sync(full, r.maxinf);
  if (lane == 0) {
    s_min[warp] = r.minfin;
    s_max[warp] = r.maxfin;
    s_ni[warp] = r.mininf;
    s_xi[warp] = r.maxinf;
  }
  __syncthreads();
  r.minfin = s_min[0];
  r.maxfin = s_max[0];
  r.mininf = s_ni[0];
  r.maxinf = s_xi[0];
#pragma unroll
  for (int w = 1; w < kNaWarps; ++w) {
    r.minfin += s_min[w];
    r.maxfin += s_max[w];
    r.mininf += s_ni[w];
    r.maxinf += s_xi[w];
  }
  __syncthreads();  // the sums are reused by the block's next row
  if (threadIdx.x == 0) na_step2(A, r);
  if (r.mininf > 1 && r.maxinf > 1) return;
  for (int64_t k = b + threadIdx.x; k < e; k += kNaThreads * kNaUnroll) {
    na_load(A, k, kNaThreads, e, a, j, L, U);
#pragma unroll
    for (int u = 0; u < kNaUnroll; ++u)
      if (k + u * kNaThreads < e) na_candidates(A, r, a[u], j[u], L[u], U[u]);
  }
}

// One round, `per` rows (32..kNaThreads, a multiple of 32) per block.  Few
// rows are spread over as many blocks as there are, since the lanes' binary64
// work shares one pipe per scheduler.  What bounds a round is the latency of
// the walks: rows of up to kNaLaneRow nonzeros go by a lane each, longer ones by
// a warp and the longest by the block, one after the other, where that is shorter
// than the longest one's walk by a lane (a row of 12,000 nonzeros takes 12 ms by
// a lane, 30 us by the block; but 32 rows of 36 in a warp's turn 210 us by the
// warp, 86 by the lanes).  A row of up to kNaWarpRow nonzeros is one FMA chain
// in CSR order whichever way it goes.
__global__ void __launch_bounds__(kNaThreads, kNaBlocksPerSM)
k_na_round(int32_t m, int per, const int64_t *row_ptr, const double *lhs_in,
           const double *rhs_in, NaArgs A) {
  const unsigned full = 0xFFFFFFFFu;
  __shared__ int s_long[kNaThreads];
  __shared__ int s_count;
  __shared__ unsigned s_rest;
  __shared__ unsigned long long s_cost, s_top;
  const int64_t i = blockIdx.x * (int64_t)per + threadIdx.x;
  NaRow r;
  r.minfin = r.maxfin = r.lhs = r.rhs = 0.0;
  r.mininf = r.maxinf = 0;
  int64_t b = 0, e = 0;
  const bool have = i < m && (int)threadIdx.x < per;
  if (have) {
    r.lhs = side_norm(lhs_in[i], A.thr);
    r.rhs = side_norm(rhs_in[i], A.thr);
    b = row_ptr[i];
    e = row_ptr[i + 1];
  }
  const unsigned long long len = (unsigned long long)(e - b);
  const bool is_long = len > kNaWarpRow;
  bool by_block = false;  // the block takes its long rows one after the other
  if (__syncthreads_or(is_long)) {
    if (threadIdx.x == 0) {
      s_count = 0;
      s_rest = 0u;
      s_cost = s_top = 0ull;
    }
    __syncthreads();
    if (is_long) {
      s_long[atomicAdd(&s_count, 1)] = threadIdx.x;
      atomicAdd(&s_cost, kNaBlockCost + len / kNaBlockShare);
      atomicMax(&s_top, len);
    }
    const unsigned most = __reduce_max_sync(full, is_long ? 0u : (unsigned)len);
    if ((threadIdx.x & 31) == 0) atomicMax(&s_rest, most);
    __syncthreads();
    // else they lengthen the lanes' walk
    by_block = s_cost < kNaLaneCost * (s_top - s_rest);
  }
  // the rows left to this warp: the mid ones by the warp one after the other, or
  // by a lane each like the others
  const unsigned wlen = is_long && by_block ? 0u : (unsigned)min(len, 1ull << 26);
  const bool mid = len > kNaLaneRow && !is_long;
  const unsigned rest = __reduce_max_sync(full, mid ? 0u : wlen);
  const bool by_warp = kNaLaneCost * rest + __reduce_add_sync(full, mid ? kNaWarpCost + 2u * wlen : 0u) <
                       kNaLaneCost * __reduce_max_sync(full, wlen);
  if (have && !(mid && by_warp) && !(is_long && by_block)) na_row_lane(A, r, b, e);
  __syncwarp();
  unsigned todo = __ballot_sync(full, mid && by_warp);
  for (; todo != 0u; todo &= todo - 1u) {
    const int src = __ffs(todo) - 1;
    NaRow q;
    q.minfin = q.maxfin = 0.0;
    q.mininf = q.maxinf = 0;
    q.lhs = __shfl_sync(full, r.lhs, src);
    q.rhs = __shfl_sync(full, r.rhs, src);
    na_row_warp(A, q, __shfl_sync(full, b, src), __shfl_sync(full, e, src));
  }
  if (!by_block) return;  // block-uniform
  __syncthreads();
  const int nlong = s_count;
  for (int q = 0; q < nlong; ++q) {  // block-uniform
    const int64_t row = blockIdx.x * (int64_t)per + s_long[q];
    NaRow x;
    x.minfin = x.maxfin = 0.0;
    x.mininf = x.maxinf = 0;
    x.lhs = side_norm(lhs_in[row], A.thr);
    x.rhs = side_norm(rhs_in[row], A.thr);
    na_row_block(A, x, row_ptr[row], row_ptr[row + 1]);
  }
}

// Ends a round: the keys become the state; crossing bounds are infeasible.
__global__ void k_na_finish(int32_t n, const uint8_t *vt, const long long *keys, double *lo,
                            double *hi, NoallocCtrl *ctrl, double eps_feas) {
  const int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (j >= n) return;
  const double L = okey_val(keys[2 * j]), U = okey_val(keys[2 * j + 1]);
  const bool cross = vt[j] ? (L > U) : (L > U + eps_feas * fmax(1.0, fabs(U)));
  if (cross) atomicExch(&ctrl->infeasible, 1);
  lo[j] = L;
  hi[j] = U;
}

// Device memory that `device` can read without peer access: memory allocated
// on that device, or managed memory.  A pointer to another GPU's memory is
// refused (reading it would need peer access the library never enables).
bool on_device(const void *p, int device) {
  if (!p) return false;
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  if (a.type == cudaMemoryTypeManaged) return true;
  return a.type == cudaMemoryTypeDevice && a.device == device;
}

// Device address of the scratch array on `device` (which must be current);
// looked up once per device.
long long *scratch_on(int device) {
  if (device < 0 || device >= kMaxDevices) return nullptr;
  long long *addr = g_scratch_addr[device].load(std::memory_order_acquire);
  if (!addr) {
    void *p = nullptr;
    if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess) {
      cudaGetLastError();
      return nullptr;
    }
    addr = static_cast<long long *>(p);
    g_scratch_addr[device].store(addr, std::memory_order_release);
  }
  return addr;
}

// Makes `device` current for its lifetime and gives the caller's current
// device back on every return path.
struct DeviceGuard {
  int prev = -1;
  bool ok = false;
  explicit DeviceGuard(int device) {
    if (cudaGetDevice(&prev) != cudaSuccess) {
      cudaGetLastError();
      prev = -1;
    }
    ok = cudaSetDevice(device) == cudaSuccess;
    if (!ok) cudaGetLastError();
  }
  ~DeviceGuard() {
    if (prev >= 0) cudaSetDevice(prev);
  }
};

int grid(int64_t work, int threads) {
  int64_t b = (work + threads - 1) / threads;
  if (b < 1) b = 1;
  if (b > 4096) b = 4096;
  return (int)b;
}

}  // namespace

extern "C" int dp_propagate_noalloc(int device, void *cuda_stream, int32_t m, int32_t n,
                                    int64_t nnz, const int64_t *row_ptr,
                                    const int32_t *col_idx, const double *val,
                                    const double *lb, const double *ub,
                                    const uint8_t *vartype, const double *lhs,
                                    const double *rhs, const dp_params *params,
                                    double *lb_out, double *ub_out, int32_t *infeasible,
                                    int32_t *rounds) {
  dp::TraceRange trace_range("dp_propagate_noalloc");
  if (!infeasible || !rounds || m < 0 || n < 0 || nnz < 0) return DP_ERR_INVALID_ARG;
  if (n > DP_NOALLOC_MAX_VARS) return DP_ERR_INVALID_ARG;
  dp_params p;
  if (params) {
    p = *params;
  } else {
    std::memset(&p, 0, sizeof(p));
    p.max_rounds = 100;
    p.eps_int = 1e-6;
    p.tau_rel = 1e-6;
    p.eps_feas = 1e-6;
    p.inf_threshold = 1e20;
  }
  if (p.max_rounds < 0 || !(p.eps_int >= 0) || !(p.tau_rel >= 0) || !(p.eps_feas >= 0) ||
      !(p.inf_threshold > 0))
    return DP_ERR_INVALID_ARG;
  DeviceGuard guard(device);
  if (!guard.ok) return DP_ERR_INVALID_ARG;
  auto dev_ok = [device](const void *q) { return on_device(q, device); };
  if (!dev_ok(row_ptr) || (nnz > 0 && (!dev_ok(col_idx) || !dev_ok(val))))
    return DP_ERR_INVALID_ARG;
  if (n > 0 && (!dev_ok(lb) || !dev_ok(ub) || !dev_ok(vartype) || !dev_ok(lb_out) ||
                !dev_ok(ub_out)))
    return DP_ERR_INVALID_ARG;
  if (m > 0 && (!dev_ok(lhs) || !dev_ok(rhs))) return DP_ERR_INVALID_ARG;
  long long *scratch = scratch_on(device);
  if (!scratch) return DP_ERR_CUDA;
  long long *keys = scratch;
  NoallocCtrl *ctrl = reinterpret_cast<NoallocCtrl *>(scratch + 2 * (size_t)DP_NOALLOC_MAX_VARS);
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);

  NoallocCtrl h;
  std::memset(&h, 0, sizeof(h));
  // the control block starts at zero on every call
  if (cudaMemsetAsync(ctrl, 0, sizeof(NoallocCtrl), st) != cudaSuccess) return DP_ERR_CUDA;
  int64_t work = nnz > (int64_t)n ? nnz : (int64_t)n;
  if ((int64_t)m + 1 > work) work = (int64_t)m + 1;
  k_na_prologue<<<grid(work, 256), 256, 0, st>>>(m, n, row_ptr, col_idx, val, nnz, lb, ub,
                                                 vartype, lhs, rhs, p.eps_int, p.inf_threshold,
                                                 lb_out, ub_out, keys, ctrl);
  if (cudaGetLastError() != cudaSuccess) return DP_ERR_CUDA;
  if (cudaMemcpyAsync(&h, ctrl, sizeof(h), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess)
    return DP_ERR_CUDA;
  if (h.err) return h.err;

  NaArgs A{};
  A.col = col_idx;
  A.val = val;
  A.vt = vartype;
  A.lo = lb_out;
  A.hi = ub_out;
  A.keys = keys;
  A.ctrl = ctrl;
  A.eps_int = p.eps_int;
  A.tau = p.tau_rel;
  A.eps_feas = p.eps_feas;
  A.thr = p.inf_threshold;
  // rows per block: as few as leave every block resident at once.  A second wave
  // of a few blocks costs as much as the first: 16k short rows in 511 blocks of
  // 32 rows 1392 us per call, in 256 of 64 rows 955; 60k irregular ones in 469
  // blocks 5278, in 235 4375.
  int sms = 1, per = 32;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess)
    return DP_ERR_CUDA;
  while (per < kNaThreads && m > (int64_t)kNaBlocksPerSM * sms * per) per *= 2;
  int32_t r = 0;
  bool changed = false;
  for (; r < p.max_rounds;) {
    if (cudaMemsetAsync(ctrl, 0, sizeof(NoallocCtrl), st) != cudaSuccess) return DP_ERR_CUDA;
    if (m > 0)
      k_na_round<<<(int)(((int64_t)m + per - 1) / per), kNaThreads, 0, st>>>(m, per, row_ptr, lhs,
                                                                            rhs, A);
    if (n > 0)
      k_na_finish<<<(int)((n + 255) / 256), 256, 0, st>>>(n, vartype, keys, lb_out, ub_out, ctrl,
                                                          p.eps_feas);
    if (cudaGetLastError() != cudaSuccess) return DP_ERR_CUDA;
    if (cudaMemcpyAsync(&h, ctrl, sizeof(h), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
      return DP_ERR_CUDA;
    ++r;
    changed = h.changed != 0;
    if (h.infeasible || !changed) break;
  }
  *rounds = r;
  *infeasible = h.infeasible ? 1 : 0;
  if (!h.infeasible && changed && r >= p.max_rounds && p.max_rounds > 0) return DP_CAP_HIT;
  return DP_OK;
}
