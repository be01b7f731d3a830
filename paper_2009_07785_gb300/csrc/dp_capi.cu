// C ABI of libdomprop.so (declared in include/domprop.h).
//
// One dp_propagate call: inputs are copied (host) or read in place (device)
// by a prologue kernel that normalises them into the matrix's workspace;
// then a CUDA graph runs the propagation rounds of Alg. 2 (arXiv 2009.07785)
// under a WHILE conditional node whose condition the last kernel of each
// round sets on the device (the role of the paper's gpu_loop, Sec. 3.7,
// without a one-thread driver kernel); an epilogue decodes the bounds; the
// stream is synchronised once.
#include <cuda_runtime.h>
#include <atomic>
#include <cstdint>
#include <cstdio>
#include <algorithm>
#include <cstring>
#include <new>
#include <vector>

#include "dp_internal.h"
#include "dp_launch.h"
#include "dp_objects.h"
#include "../../include/domprop.h"
#include "dp_trace.h"

namespace dp {
namespace {
std::atomic<int32_t> g_fail_countdown{0};  // the k-th allocation from now fails (0: none)
std::atomic<int64_t> g_live_allocs{0};
}  // namespace

cudaError_t dev_malloc(void **p, size_t bytes) {
  int32_t k = g_fail_countdown.load();
  while (k > 0 && !g_fail_countdown.compare_exchange_weak(k, k - 1)) {
  }
  if (k == 1) {  // this allocation is the one asked to fail
    *p = nullptr;
    return cudaErrorMemoryAllocation;
  }
  const cudaError_t e = cudaMalloc(p, bytes);
  if (e == cudaSuccess) g_live_allocs.fetch_add(1);
  return e;
}

void dev_free(void *p) {
  if (!p) return;
  cudaFree(p);
  g_live_allocs.fetch_sub(1);
}

void arm_alloc_failure(int32_t k) { g_fail_countdown.store(k); }
int64_t live_allocs() { return g_live_allocs.load(); }
}  // namespace dp

namespace {

#define CUDA_TRY(x)                          \
  do {                                       \
    cudaError_t e_ = (x);                    \
    if (e_ != cudaSuccess) return DP_ERR_CUDA; \
  } while (0)

template <typename T>
int dev_alloc(dp_matrix *mat, T **p, size_t count) {
  void *q = nullptr;
  size_t bytes = sizeof(T) * (count > 0 ? count : 1);
  cudaError_t e = dp::dev_malloc(&q, bytes);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return e == cudaErrorMemoryAllocation ? DP_ERR_OOM : DP_ERR_CUDA;
  }
  mat->allocs.push_back(q);
  *p = static_cast<T *>(q);
  return DP_OK;
}

template <typename T>
int upload(dp_matrix *mat, const std::vector<T> &v, const T **out, cudaStream_t st) {
  T *d = nullptr;
  int rc = dev_alloc(mat, &d, v.size());
  if (rc) return rc;
  if (!v.empty()) CUDA_TRY(cudaMemcpyAsync(d, v.data(), sizeof(T) * v.size(), cudaMemcpyHostToDevice, st));
  *out = d;
  return DP_OK;
}

using dp::is_device_ptr;

// A round that is expected to change more than n / kMarkShare variables does
// not mark their chunks, and the next one processes all of them: marking costs
// an atomic per nonzero of the changed variables, and at that share every long
// row is marked anyway.
constexpr int32_t kMarkShare = 32;

// Where a team (dp_team.cu) takes a problem instead of the graph's kernels or
// the batched ones.  A team's rounds cost less (a cluster barrier instead of
// three to five kernels) and its marking skips unchanged rows, but it has 16
// blocks at most.  Measured in us per call (graph or batch / team), both in one
// run of the same build:
//   one problem:  short rows 50k nonzeros 542 / 405, 100k 605 / 582, 140k 533 / 681;
//                 irregular 55k 832 / 749, 110k 853 / 781, 226k 1187 / 1318;
//                 mixed 42k 1185 / 865, 80k 1036 / 1068, 116k 1375 / 1620;
//                 90k in rows of 3 (938 slices) 346 / 458, of 6 (470) 510 / 497
//   nodes:        irregular 60k nonzeros, 8 nodes 1521 / 772 in many rounds and 171 /
//                 127 in one, 33 nodes 2221 / 1151 and 190 / 199, 100 nodes
//                 2621 / 2166; 90k, 33 nodes 7981 / 2256 and 210 / 236; 140k, 8
//                 nodes 3235 / 1269 and 171 / 204; 250k, 1 node 2928 / 1573 and 175 /
//                 226, 16 nodes 3267 / 2933;
//                 short rows 60k, 8 nodes 734 / 472, 33 nodes 953 / 672, 100 nodes
//                 1369 / 1622; 90k, 12 nodes 780 / 611 (3.7 slices per warp), 16
//                 nodes 764 / 811 (7.3);
//                 1000 nodes over 2k in rows of 6 1545 / 927 (10 items), of 30 387 /
//                 712 (34 items); over 4k in rows of 4 2372 / 1824 (31 items), over 12k in
//                 rows of 6 2274 / 2837 (63 items)
//   sets:         64 problems of 300 rows 770 / 352, 64 of up to 60,000 2727 / 6348;
//                 1000 of 300 1961 / 1248; 8000 of 20 3892 / 3857, of 100 4967 /
//                 4803; 10,000 of 20 4229 / 4738, 20,000 of 20 6701 / 8761, of 10
//                 5696 / 5474, of 2 3255 / 2134; 50,000 of 2 3481 / 4405, 100,000 of 1
//                 1247 / 6621
constexpr int64_t kTeamNnz = 100000;       // a single problem, a set's largest, a node
                                           // batch's matrix without long slices
constexpr int32_t kTeamSlices = 640;       // slices of a single problem
constexpr int64_t kTeamSetNnz = 4000000;   // a whole set
constexpr int32_t kTeamSetCount = 8192;    // its problems; three times as many
constexpr int64_t kTeamSetFew = 1000000;   // if they have this many nonzeros or fewer
constexpr int64_t kTeamSetPad = 24;        // its slots per nonzero
constexpr int64_t kTeamNodeNnz = 300000;   // the matrix of a node batch with long slices
constexpr int64_t kTeamNodeWork = 2500000;  // nonzeros times nodes: up to kTeamNnz nonzeros,
constexpr int64_t kTeamNodeWorkLong = 1000000;  // and above
constexpr int64_t kTeamNodeItems = 32;     // team_items of a matrix with more nodes than teams
constexpr int64_t kTeamNodeShare = 6;      // team_items per warp without long slices
constexpr int kTeamWarps = 8;  // warps per block of a team

// What the warps of a team share out in a round: the slices, the long ones
// chunk by chunk.
int64_t team_items(int32_t nslices, int32_t nlong) {
  return nslices + (int64_t)(dp::kSliceW - 1) * nlong;
}

// Blocks of a team, a power of two: no more than give every item a warp and
// all `count` teams room at once.  (With a warp per slice 100 rows of 200
// nonzeros had one block: 691 us per call, with 16 blocks 197.)
int team_size(const dp_ctx *ctx, int64_t items, int32_t count) {
  int k = 4;
  while (k > 0 && ((1 << k) > 2 * ((items + kTeamWarps - 1) / kTeamWarps) - 1 ||
                   ctx->teams_of[k] < count))
    --k;
  return k;  // log2
}

// The parameters of a call.
void team_params(dp::TeamArgs &A, const dp_params &p) {
  A.max_rounds = p.max_rounds;
  A.eps_int = p.eps_int;
  A.tau_rel = p.tau_rel;
  A.eps_feas = p.eps_feas;
  A.inf_thr = p.inf_threshold;
}

// Makes a round-loop graph: one WHILE node whose body is the kernels that
// `body(handle, stream)` launches; the condition starts at 1 on every launch
// and the last kernel of the body sets it on the device.
template <typename Body>
int build_loop_graph(Body body, cudaGraph_t *graph_out, cudaGraphExec_t *exec_out) {
  cudaGraph_t g = nullptr;
  CUDA_TRY(cudaGraphCreate(&g, 0));
  cudaGraphConditionalHandle h;
  if (cudaGraphConditionalHandleCreate(&h, g, 1, cudaGraphCondAssignDefault) != cudaSuccess) {
    cudaGraphDestroy(g);
    return DP_ERR_CUDA;
  }
  cudaGraphNodeParams np = {cudaGraphNodeTypeConditional};
  np.conditional.handle = h;
  np.conditional.type = cudaGraphCondTypeWhile;
  np.conditional.size = 1;
  cudaGraphNode_t node;
  if (cudaGraphAddNode(&node, g, nullptr, nullptr, 0, &np) != cudaSuccess) {
    cudaGraphDestroy(g);
    return DP_ERR_CUDA;
  }
  cudaGraph_t bodyg = np.conditional.phGraph_out[0];
  cudaStream_t cs = nullptr;
  if (cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking) != cudaSuccess) {
    cudaGraphDestroy(g);
    return DP_ERR_CUDA;
  }
  cudaError_t e = cudaStreamBeginCaptureToGraph(cs, bodyg, nullptr, nullptr, 0,
                                                cudaStreamCaptureModeRelaxed);
  if (e == cudaSuccess) {
    cudaError_t le = body(h, cs);
    cudaGraph_t captured = nullptr;
    e = cudaStreamEndCapture(cs, &captured);
    if (le != cudaSuccess) e = le;
  }
  cudaStreamDestroy(cs);
  if (e != cudaSuccess) {
    cudaGetLastError();
    cudaGraphDestroy(g);
    return DP_ERR_CUDA;
  }
  cudaGraphExec_t ex = nullptr;
  if (cudaGraphInstantiate(&ex, g, 0) != cudaSuccess) {
    cudaGetLastError();
    cudaGraphDestroy(g);
    return DP_ERR_CUDA;
  }
  *graph_out = g;
  *exec_out = ex;
  return DP_OK;
}

// The variables' records are gathered once per nonzero and round while the
// matrix streams past them; the round graph's kernels ask L2 to keep the
// records resident (an access-policy window with the persisting property,
// within the L2 set-aside of this context) so that the stream does not
// evict them.  Best effort: a device or driver that refuses leaves the
// ordinary policy in place.
void l2_keep_records(const dp_matrix *mat, cudaStream_t cs) {
  const size_t bytes = sizeof(dp::VarRec) * (size_t)(mat->M.n > 0 ? mat->M.n : 1);
  int max_persist = 0, max_window = 0;
  const int dev = mat->ctx->device;
  if (cudaDeviceGetAttribute(&max_persist, cudaDevAttrMaxPersistingL2CacheSize, dev) !=
          cudaSuccess ||
      cudaDeviceGetAttribute(&max_window, cudaDevAttrMaxAccessPolicyWindowSize, dev) !=
          cudaSuccess ||
      max_persist <= 0 || max_window <= 0) {
    cudaGetLastError();
    return;
  }
  size_t cur = 0;
  cudaDeviceGetLimit(&cur, cudaLimitPersistingL2CacheSize);
  const size_t want = bytes < (size_t)max_persist ? bytes : (size_t)max_persist;
  if (cur < want && cudaDeviceSetLimit(cudaLimitPersistingL2CacheSize, want) != cudaSuccess) {
    cudaGetLastError();
    return;
  }
  cudaDeviceGetLimit(&cur, cudaLimitPersistingL2CacheSize);
  cudaStreamAttrValue v = {};
  v.accessPolicyWindow.base_ptr = mat->S.rec;
  v.accessPolicyWindow.num_bytes = bytes < (size_t)max_window ? bytes : (size_t)max_window;
  const double ratio = (double)cur / (double)v.accessPolicyWindow.num_bytes;
  v.accessPolicyWindow.hitRatio = (float)(ratio < 1.0 ? ratio : 1.0);
  v.accessPolicyWindow.hitProp = cudaAccessPropertyPersisting;
  v.accessPolicyWindow.missProp = cudaAccessPropertyStreaming;
  if (cudaStreamSetAttribute(cs, cudaStreamAttributeAccessPolicyWindow, &v) != cudaSuccess)
    cudaGetLastError();
}

int build_graph(dp_matrix *mat) {
  const int sms = mat->ctx->num_sms;
  return build_loop_graph(
      [mat, sms](cudaGraphConditionalHandle h, cudaStream_t cs) {
        l2_keep_records(mat, cs);
        return dp::launch_round_body(mat->M, mat->S, mat->vt_ws, h, sms, cs);
      },
      &mat->graph, &mat->exec);
}

}  // namespace

extern "C" {

int dp_params_default(dp_params *out) {
  if (!out) return DP_ERR_INVALID_ARG;
  std::memset(out, 0, sizeof(*out));
  out->max_rounds = 100;
  out->eps_int = 1e-6;
  out->tau_rel = 1e-6;
  out->eps_feas = 1e-6;
  out->inf_threshold = 1e20;
  return DP_OK;
}

const char *dp_strerror(int code) {
  switch (code) {
    case DP_OK: return "ok";
    case DP_CAP_HIT: return "round cap hit (bounds valid)";
    case DP_ERR_INVALID_ARG: return "invalid argument";
    case DP_ERR_BAD_CSR: return "malformed CSR matrix or invalid coefficient";
    case DP_ERR_NAN_INPUT: return "NaN or contradictory infinity in bounds or sides";
    case DP_ERR_OOM: return "out of memory";
    case DP_ERR_CUDA: return "CUDA runtime error";
    case DP_ERR_TIMEOUT: return "bounded device wait timed out";
    default: return "unknown status";
  }
}

int dp_ctx_set_wait_limit(dp_ctx *ctx, int64_t sleeps) {
  if (!ctx || sleeps < 0) return DP_ERR_INVALID_ARG;
  ctx->wait_limit = sleeps == 0 ? dp::kDefaultWaitLimit : (long long)sleeps;
  return DP_OK;
}

int dp_debug_fail_alloc(int32_t k) {
  if (k < 0) return DP_ERR_INVALID_ARG;
  dp::arm_alloc_failure(k);
  return DP_OK;
}

int64_t dp_debug_live_allocs(void) { return dp::live_allocs(); }

int dp_create(dp_ctx **out, int device, void *cuda_stream) {
  if (!out) return DP_ERR_INVALID_ARG;
  *out = nullptr;
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess) {
    cudaGetLastError();
    return DP_ERR_CUDA;
  }
  if (device < 0 || device >= ndev) return DP_ERR_INVALID_ARG;
  CUDA_TRY(cudaSetDevice(device));
  dp_ctx *ctx = new (std::nothrow) dp_ctx();
  if (!ctx) return DP_ERR_OOM;
  ctx->device = device;
  if (cudaDeviceGetAttribute(&ctx->num_sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess) {
    delete ctx;
    return DP_ERR_CUDA;
  }
  for (int k = 0; k < 5; ++k) ctx->teams_of[k] = dp::cluster_teams_resident(1 << k);
  if (cuda_stream) {
    ctx->stream = static_cast<cudaStream_t>(cuda_stream);
  } else {
    if (cudaStreamCreateWithFlags(&ctx->stream, cudaStreamNonBlocking) != cudaSuccess) {
      delete ctx;
      return DP_ERR_CUDA;
    }
    ctx->own_stream = true;
  }
  // the results of teams first (16-byte aligned), the control block behind
  if (cudaMallocHost(&ctx->h_res, sizeof(int4) + sizeof(dp::Ctrl)) != cudaSuccess) {
    if (ctx->own_stream) cudaStreamDestroy(ctx->stream);
    delete ctx;
    return DP_ERR_OOM;
  }
  ctx->h_ctrl = reinterpret_cast<dp::Ctrl *>(ctx->h_res + 1);
  *out = ctx;
  return DP_OK;
}

void dp_destroy(dp_ctx *ctx) {
  if (!ctx) return;
  cudaSetDevice(ctx->device);
  if (ctx->h_res) cudaFreeHost(ctx->h_res);
  if (ctx->own_stream) cudaStreamDestroy(ctx->stream);
  delete ctx;
}

namespace {
void free_batch(BatchWs *b) {
  if (!b) return;
  for (int k = 0; k < dp::kActKinds; ++k) {
    if (b->exec[k]) cudaGraphExecDestroy(b->exec[k]);
    if (b->graph[k]) cudaGraphDestroy(b->graph[k]);
  }
  for (void *p : b->allocs) dp::dev_free(p);
  if (b->h_ctrl) cudaFreeHost(b->h_ctrl);
  if (b->h_nodes) cudaFreeHost(b->h_nodes);
  delete b;
}

void free_teams(TeamWs *t) {
  if (!t) return;
  for (void *p : t->allocs) dp::dev_free(p);
  dp::dev_free(t->st_lb);
  dp::dev_free(t->st_ub);
  dp::dev_free(t->out_lb);
  dp::dev_free(t->out_ub);
  if (t->h_res) cudaFreeHost(t->h_res);
  delete t;
}
}  // namespace

void dp_matrix_free(dp_matrix *mat) {
  if (!mat) return;
  cudaSetDevice(mat->ctx->device);
  cudaStreamSynchronize(mat->ctx->stream);
  free_batch(mat->batch);
  free_teams(mat->teams);
  if (mat->h_inst) cudaFreeHost(mat->h_res);  // a set's; else the context's
  if (mat->exec) cudaGraphExecDestroy(mat->exec);
  if (mat->graph) cudaGraphDestroy(mat->graph);
  for (void *p : mat->allocs) dp::dev_free(p);
  mat->ctx->live_matrices--;
  delete mat;
}

int dp_matrix_load(dp_ctx *ctx, int32_t m, int32_t n, int64_t nnz,
                   const int64_t *row_ptr, const int32_t *col_idx,
                   const double *val, int32_t chunk, dp_matrix **out) {
  dp::TraceRange trace_range("dp_matrix_load");
  return dp_matrix_load_sides(ctx, m, n, nnz, row_ptr, col_idx, val, chunk, nullptr, nullptr,
                              out);
}

}  // extern "C"

namespace {

// Loads a matrix from its host layout; with row_off/var_off (count+1 offsets
// each) it is the block-diagonal union of `count` independent problems; with
// `views` (largest first) it was laid out problem by problem.
int load_layout(dp_ctx *ctx, dp::HostLayout &H, const std::vector<int32_t> *row_off,
                const std::vector<int32_t> *var_off, const std::vector<dp::TeamView> *views,
                dp_matrix **out) {
  const int32_t m = H.m, n = H.n;
  const int64_t nnz = H.nnz;
  CUDA_TRY(cudaSetDevice(ctx->device));
  dp_matrix *mat = new (std::nothrow) dp_matrix();
  if (!mat) return DP_ERR_OOM;
  mat->ctx = ctx;
  ctx->live_matrices++;
  cudaStream_t st = ctx->stream;
  dp::DevMatrix &M = mat->M;
  M.m = m;
  M.n = n;
  M.nnz = nnz;
  M.nslices = H.nslices;
  M.nslices_split = H.nslices_split;
  M.nsplit_rows = H.nsplit_rows;
  M.round_warps = 8;
  M.layout = H.layout;
  M.mp_ipt = H.mp_ipt;
  M.mp_nseg = H.mp_nseg;
  M.mp_nlong = H.mp_nlong;
  M.mp_npiece = (int32_t)H.mp_piece.size();
  // the order in which a round takes the slices, and the candidate queues' room: the
  // slots of their slices (merge path: the nonzeros of every 32 rows in the
  // layout's order)
  std::vector<int32_t> order;
  std::vector<uint32_t> qbase;
  M.short0 = H.nslices;
  try {
    if (H.layout == dp::kLayoutEll) {
      auto len = [&](int32_t q) { return H.slice_len[(size_t)q]; };
      auto is_short = [&](int32_t q) { return q >= H.nslices_split && len(q) <= dp::kShortRow; };
      for (int32_t q = 0; q < H.nslices; ++q) {
        M.nlong += len(q) >= dp::kLongSlots;
        M.max_slots = std::max(M.max_slots, len(q));
      }
      if (views) {
        order.resize((size_t)H.nslices);
        for (int32_t q = 0; q < H.nslices; ++q) order[(size_t)q] = q;
        std::stable_sort(order.begin(), order.end(), [&](int32_t x, int32_t y) {
          return is_short(x) != is_short(y) ? is_short(y) : len(x) > len(y);
        });
        while (M.short0 > 0 && is_short(order[(size_t)M.short0 - 1])) --M.short0;
      } else {  // both kinds of slices are sorted, longest first
        while (M.long_split < M.nslices_split && len(M.long_split) >= dp::kLongSlots) ++M.long_split;
        M.long_whole = M.nlong - M.long_split;
        while (M.short0 > 0 && is_short(M.short0 - 1)) --M.short0;
      }
    }
    std::vector<int64_t> room(dp::kQueues, 0);
    for (int32_t q = 0; q < H.nslices; ++q)
      for (int t = 0; t < dp::kSliceW; ++t)
        room[(size_t)(q % dp::kQueues)] +=
            H.chunk_len[(size_t)q * dp::kSliceW + (size_t)t] & dp::kLenMask;
    qbase.assign(dp::kQueues, 0);
    for (size_t q = 1; q < qbase.size(); ++q)
      qbase[q] = (uint32_t)(qbase[q - 1] + room[q - 1]);
    if (row_off) {
      mat->row_off = *row_off;
      mat->var_off = *var_off;
    }
  } catch (const std::bad_alloc &) {
    dp_matrix_free(mat);
    return DP_ERR_OOM;
  }
  mat->padded = (int64_t)H.val.size();
#define TRY(x)                 \
  do {                         \
    int r_ = (x);              \
    if (r_) {                  \
      dp_matrix_free(mat);     \
      return r_;               \
    }                          \
  } while (0)
  TRY(upload(mat, H.val, &M.val, st));
  if (!H.val8.empty()) {
    TRY(upload(mat, H.val8, &mat->val8, st));
    M.val8 = nullptr;  // off by default: measured slower on GB300 (see the header)
  }
  TRY(upload(mat, H.col, &M.col, st));
  TRY(upload(mat, H.slice_off, &M.slice_off, st));
  TRY(upload(mat, H.slice_len, &M.slice_len, st));
  if (!order.empty()) TRY(upload(mat, order, &M.order, st));
  TRY(upload(mat, H.chunk_row, &M.chunk_row, st));
  TRY(upload(mat, H.chunk_len, &M.chunk_len, st));
  TRY(upload(mat, H.chunk_sidx, &M.chunk_sidx, st));
  TRY(upload(mat, H.split_row, &M.split_row, st));
  TRY(upload(mat, H.split_cbeg, &M.split_cbeg, st));
  TRY(upload(mat, H.split_cidx, &M.split_cidx, st));
  TRY(upload(mat, H.mp_ptr, &M.mp_ptr, st));
  TRY(upload(mat, H.mp_srow, &M.mp_srow, st));
  TRY(upload(mat, H.mp_piece, &M.mp_piece, st));
  dp::DevState &S = mat->S;
  TRY(dev_alloc(mat, &S.rec, (size_t)n));
  TRY(dev_alloc(mat, &S.keys, 2 * (size_t)n));
  TRY(dev_alloc(mat, &S.lhs, (size_t)m));
  TRY(dev_alloc(mat, &S.rhs, (size_t)m));
  if (H.layout == dp::kLayoutMerge) {
    // pieces: head and carry of every segment; activities of every row
    TRY(dev_alloc(mat, &S.part, 2 * (size_t)H.mp_nseg));
    TRY(dev_alloc(mat, &S.rowact, (size_t)m));
    TRY(dev_alloc(mat, &S.mp_need, ((size_t)H.mp_nseg + 31) / 32));
    TRY(dev_alloc(mat, &S.rowtot, (size_t)H.mp_nlong));
  } else {
    TRY(dev_alloc(mat, &S.part, (size_t)H.nslices_split * dp::kSliceW));
    TRY(dev_alloc(mat, &S.rowtot, (size_t)H.nsplit_rows));
  }
  // candidate queue: at most one entry per slot and round, so it never
  // overflows; row sums are stored per chunk slot
  TRY(dev_alloc(mat, &S.queue, (size_t)mat->padded));
  TRY(upload(mat, qbase, &S.qbase, st));
  TRY(dev_alloc(mat, &S.qcount, (size_t)dp::kQueues * dp::kQueueStep));
  if (cudaMemsetAsync(S.qcount, 0, sizeof(int32_t) * dp::kQueues * dp::kQueueStep, st) !=
      cudaSuccess) {
    cudaGetLastError();
    dp_matrix_free(mat);
    return DP_ERR_CUDA;
  }
  TRY(dev_alloc(mat, &S.rowsum, (size_t)H.nslices * dp::kSliceW));
  TRY(dev_alloc(mat, &S.side, (size_t)H.nslices * dp::kSliceW));
  TRY(dev_alloc(mat, &S.ctrl, 1));
  // dirty bitmap (a set's problems start at words of their own when teams run)
  TRY(dev_alloc(mat, &S.dirty, ((size_t)n + 31) / 32 + (views ? views->size() : 0)));
  TRY(dev_alloc(mat, &S.bar, 2));
  if (H.layout == dp::kLayoutEll) {
    int32_t *ptr = nullptr, *slot = nullptr;
    TRY(dev_alloc(mat, &ptr, (size_t)n + 1));
    TRY(dev_alloc(mat, &slot, (size_t)nnz));
    const size_t nflags = views ? views->size() : 1;
    TRY(dev_alloc(mat, &mat->team_flags, nflags));
    TRY(dev_alloc(mat, &mat->team_mask, 2 * (size_t)H.nslices));
    TRY(dev_alloc(mat, &mat->team_touch, (size_t)H.nsplit_rows));
    // the counts' scratch: the keys are not in use yet
    if (dp::launch_columns(M, reinterpret_cast<int32_t *>(S.keys), ptr, slot, ctx->num_sms, st) !=
            cudaSuccess ||
        cudaMemsetAsync(mat->team_flags, 0, sizeof(dp::TeamFlags) * nflags, st) != cudaSuccess) {
      cudaGetLastError();
      dp_matrix_free(mat);
      return DP_ERR_CUDA;
    }
    M.col_ptr = ptr;
    M.col_slot = slot;
    S.mask = mat->team_mask;  // one call on a matrix at a time
    S.touch = mat->team_touch;
    mat->h_res = ctx->h_res;
  }
  TRY(dev_alloc(mat, &mat->vt_ws, (size_t)n));
  TRY(dev_alloc(mat, &mat->st_lb, (size_t)n));
  TRY(dev_alloc(mat, &mat->st_ub, (size_t)n));
  TRY(dev_alloc(mat, &mat->st_vt, (size_t)n));
  TRY(dev_alloc(mat, &mat->st_lhs, (size_t)m));
  TRY(dev_alloc(mat, &mat->st_rhs, (size_t)m));
  TRY(dev_alloc(mat, &mat->out_lb, (size_t)n));
  TRY(dev_alloc(mat, &mat->out_ub, (size_t)n));
  if (row_off) {
    // problem of every chunk slot (by its row) and of every variable
    const int32_t count = (int32_t)row_off->size() - 1;
    std::vector<int32_t> slot_inst(H.chunk_row.size(), -1), var_inst((size_t)n, 0);
    for (size_t c = 0; c < H.chunk_row.size(); ++c) {
      const int32_t r = H.chunk_row[c];
      if (r >= 0)
        slot_inst[c] = (int32_t)(std::upper_bound(row_off->begin(), row_off->end(), r) -
                                 row_off->begin()) - 1;
    }
    for (int32_t k = 0; k < count; ++k)
      for (int32_t j = (*var_off)[k]; j < (*var_off)[k + 1]; ++j) var_inst[(size_t)j] = k;
    TRY(upload(mat, slot_inst, &S.I.slot_inst, st));
    TRY(upload(mat, var_inst, &S.I.var_inst, st));
    TRY(dev_alloc(mat, &S.I.changed, (size_t)count));
    TRY(dev_alloc(mat, &S.I.infeasible, (size_t)count));
    TRY(dev_alloc(mat, &S.I.done, (size_t)count));
    TRY(dev_alloc(mat, &S.I.rounds, (size_t)count));
    TRY(dev_alloc(mat, &S.I.status, (size_t)count));
    S.I.ninst = count;
    mat->ninst = count;
    if (views) {
      const dp::TeamView *dv = nullptr;
      TRY(upload(mat, *views, &dv, st));
      mat->d_views = const_cast<dp::TeamView *>(dv);
      TRY(dev_alloc(mat, &mat->team_next, 1));
    }
    int4 *pinned = nullptr;
    if (cudaMallocHost(&pinned, (sizeof(int4) + 3 * sizeof(int32_t)) * (size_t)count) !=
        cudaSuccess) {
      cudaGetLastError();
      dp_matrix_free(mat);
      return DP_ERR_OOM;
    }
    mat->h_res = pinned;
    mat->h_inst = reinterpret_cast<int32_t *>(pinned + count);
  }
  if (cudaStreamSynchronize(st) != cudaSuccess) {
    cudaGetLastError();
    dp_matrix_free(mat);
    return DP_ERR_CUDA;
  }
  TRY(build_graph(mat));
#undef TRY
  *out = mat;
  return DP_OK;
}

// Loads one matrix; with merge_ipt > 0 it gets the merge-path layout with
// that many items per segment.
int load_impl(dp_ctx *ctx, int32_t m, int32_t n, int64_t nnz, const int64_t *row_ptr,
              const int32_t *col_idx, const double *val, int32_t chunk, const double *lhs,
              const double *rhs, dp_matrix **out, int32_t merge_ipt = 0) {
  if (!ctx || !out) return DP_ERR_INVALID_ARG;
  *out = nullptr;
  if ((lhs == nullptr) != (rhs == nullptr)) return DP_ERR_INVALID_ARG;
  dp::HostLayout H;
  int rc = merge_ipt > 0
               ? dp::build_merge_layout(m, n, nnz, row_ptr, col_idx, val, merge_ipt, lhs, rhs, H)
               : dp::build_layout(m, n, nnz, row_ptr, col_idx, val, chunk, lhs, rhs, H);
  if (rc) return rc;
  return load_layout(ctx, H, nullptr, nullptr, nullptr, out);
}

// Whether a set is loaded problem by problem, for a team each, and not as one
// union whose rows share length-sorted slices: small problems, not too many of
// them, and no more than kTeamSetPad slots to a nonzero (every problem is padded
// to whole slices, up to 32 slots to a nonzero for problems of one row).
bool set_by_teams(const dp_ctx *ctx, int32_t count, const int32_t *m,
                  const int64_t *const *row_ptr, int64_t nnz, int32_t chunk) {
  if (ctx->teams_of[0] <= 0 || nnz > kTeamSetNnz ||
      count > (nnz <= kTeamSetFew ? 3 : 1) * kTeamSetCount)
    return false;
  if (chunk == 0) chunk = 256;
  if (chunk < 8) return false;  // refused by the layout
  int64_t slots = 0;
  std::vector<int32_t> whole, piece;
  for (int32_t k = 0; k < count; ++k) {
    whole.clear();
    piece.clear();
    if (m[k] > 0 && row_ptr[k][m[k]] > kTeamNnz) return false;
    for (int32_t i = 0; i < m[k]; ++i) {
      int64_t len = row_ptr[k][i + 1] - row_ptr[k][i];
      if (len < 0 || len > nnz) return false;  // refused by the layout
      if (len <= chunk) {
        whole.push_back((int32_t)len);
        continue;
      }
      for (; len > 0; len -= chunk) piece.push_back((int32_t)(len < chunk ? len : chunk));
    }
    for (std::vector<int32_t> *v : {&whole, &piece}) {
      std::sort(v->begin(), v->end(), [](int32_t x, int32_t y) { return x > y; });
      for (size_t q = 0; q < v->size(); q += dp::kSliceW) slots += (int64_t)dp::kSliceW * (*v)[q];
    }
  }
  return slots <= kTeamSetPad * nnz;
}

// The layout of the block-diagonal union as one matrix.
int build_union(int32_t count, const int32_t *m, const int32_t *n, const int64_t *const *row_ptr,
                const int32_t *const *col_idx, const double *const *val, int32_t chunk,
                const double *const *lhs, const double *const *rhs, int32_t rows, int64_t nnz,
                const std::vector<int32_t> &var_off, dp::HostLayout &H) {
  std::vector<int64_t> rp(1, 0);
  std::vector<int32_t> col;
  std::vector<double> vv, sl, sr;
  rp.reserve((size_t)rows + 1);
  col.reserve((size_t)std::max<int64_t>(nnz, 0));
  vv.reserve((size_t)std::max<int64_t>(nnz, 0));
  for (int32_t k = 0; k < count; ++k) {
    const int64_t base = rp.back(), nz = m[k] > 0 ? row_ptr[k][m[k]] : 0;
    for (int32_t i = 0; i < m[k]; ++i) rp.push_back(base + row_ptr[k][i + 1]);
    for (int64_t q = 0; q < nz; ++q) {
      const int32_t c = col_idx[k][q];
      if (c < 0 || c >= n[k]) return DP_ERR_BAD_CSR;
      col.push_back(c + var_off[(size_t)k]);
      vv.push_back(val[k][q]);
    }
    if (lhs) {
      sl.insert(sl.end(), lhs[k], lhs[k] + m[k]);
      sr.insert(sr.end(), rhs[k], rhs[k] + m[k]);
    }
  }
  return dp::build_layout(rows, var_off.back(), nnz, rp.data(), col.data(), vv.data(), chunk,
                          lhs ? sl.data() : nullptr, lhs ? sr.data() : nullptr, H);
}

}  // namespace

extern "C" {

int dp_matrix_load_sides(dp_ctx *ctx, int32_t m, int32_t n, int64_t nnz,
                         const int64_t *row_ptr, const int32_t *col_idx, const double *val,
                         int32_t chunk, const double *lhs, const double *rhs,
                         dp_matrix **out) {
  dp::TraceRange trace_range("dp_matrix_load_sides");
  return load_impl(ctx, m, n, nnz, row_ptr, col_idx, val, chunk, lhs, rhs, out);
}

int dp_matrix_load_merge(dp_ctx *ctx, int32_t m, int32_t n, int64_t nnz,
                         const int64_t *row_ptr, const int32_t *col_idx, const double *val,
                         int32_t items_per_thread, const double *lhs, const double *rhs,
                         dp_matrix **out) {
  dp::TraceRange trace_range("dp_matrix_load_merge");
  if (items_per_thread < 4 || items_per_thread > 4096) {
    if (out) *out = nullptr;
    return DP_ERR_INVALID_ARG;
  }
  return load_impl(ctx, m, n, nnz, row_ptr, col_idx, val, 0, lhs, rhs, out, items_per_thread);
}

int dp_matrix_load_set(dp_ctx *ctx, int32_t count, const int32_t *m, const int32_t *n,
                       const int64_t *const *row_ptr, const int32_t *const *col_idx,
                       const double *const *val, int32_t chunk, const double *const *lhs,
                       const double *const *rhs, dp_matrix **out) {
  dp::TraceRange trace_range("dp_matrix_load_set");
  if (!ctx || !out || count <= 0 || !m || !n || !row_ptr || !col_idx || !val)
    return DP_ERR_INVALID_ARG;
  *out = nullptr;
  if ((lhs == nullptr) != (rhs == nullptr)) return DP_ERR_INVALID_ARG;
  try {
    std::vector<int32_t> row_off(1, 0), var_off(1, 0);
    int64_t mt = 0, nt = 0, nzt = 0;
    for (int32_t k = 0; k < count; ++k) {
      if (m[k] < 0 || n[k] < 0 || (m[k] > 0 && !row_ptr[k])) return DP_ERR_INVALID_ARG;
      mt += m[k];
      nt += n[k];
      if (m[k] > 0) nzt += row_ptr[k][m[k]];
      if (mt >= (int64_t(1) << 31) || nt >= (int64_t(1) << 31) || nzt >= (int64_t(1) << 31))
        return DP_ERR_INVALID_ARG;
      row_off.push_back((int32_t)mt);
      var_off.push_back((int32_t)nt);
    }
    for (int32_t k = 0; k < count; ++k) {
      if (m[k] > 0 && row_ptr[k][0] != 0) return DP_ERR_BAD_CSR;
      if (m[k] > 0 && row_ptr[k][m[k]] > 0 && (!col_idx[k] || !val[k])) return DP_ERR_INVALID_ARG;
    }
    dp::HostLayout H;
    std::vector<dp::TeamView> views;
    int rc;
    if (set_by_teams(ctx, count, m, row_ptr, nzt, chunk))
      rc = dp::build_set_layout(count, m, n, row_ptr, col_idx, val, chunk, lhs, rhs, H, views);
    else
      rc = build_union(count, m, n, row_ptr, col_idx, val, chunk, lhs, rhs, (int32_t)mt, nzt,
                       var_off, H);
    if (rc) return rc;
    dp_matrix *set = nullptr;
    rc = load_layout(ctx, H, &row_off, &var_off, views.empty() ? nullptr : &views, &set);
    if (rc) return rc;
    if (!views.empty()) {
      const dp::TeamView &V = views.front();
      set->view_items =
          team_items((V.split1 - V.split0) + (V.whole1 - V.whole0), V.nlsplit + V.nlwhole);
    }
    *out = set;
    return DP_OK;
  } catch (const std::bad_alloc &) {
    return DP_ERR_OOM;
  }
}

int dp_matrix_set_launch(dp_matrix *mat, int32_t round_warps) {
  if (!mat || (round_warps != 4 && round_warps != 8)) return DP_ERR_INVALID_ARG;
  if (mat->M.round_warps == round_warps) return DP_OK;
  CUDA_TRY(cudaSetDevice(mat->ctx->device));
  CUDA_TRY(cudaStreamSynchronize(mat->ctx->stream));
  if (mat->exec) cudaGraphExecDestroy(mat->exec);
  if (mat->graph) cudaGraphDestroy(mat->graph);
  mat->exec = nullptr;
  mat->graph = nullptr;
  mat->M.round_warps = round_warps;
  return build_graph(mat);
}

int dp_matrix_set_compression(dp_matrix *mat, int32_t on, int32_t *active) {
  if (!mat) return DP_ERR_INVALID_ARG;
  const int8_t *want = (on && mat->val8) ? mat->val8 : nullptr;
  if (want != mat->M.val8) {
    CUDA_TRY(cudaSetDevice(mat->ctx->device));
    CUDA_TRY(cudaStreamSynchronize(mat->ctx->stream));
    if (mat->exec) cudaGraphExecDestroy(mat->exec);
    if (mat->graph) cudaGraphDestroy(mat->graph);
    mat->exec = nullptr;
    mat->graph = nullptr;
    mat->M.val8 = want;
    int rc = build_graph(mat);
    if (rc) return rc;
  }
  if (active) *active = mat->M.val8 ? 1 : 0;
  return DP_OK;
}

int dp_matrix_set_offsets(const dp_matrix *set, int32_t *count, int32_t *row_off,
                          int32_t *var_off) {
  if (!set) return DP_ERR_INVALID_ARG;
  if (count) *count = set->ninst;
  for (int32_t k = 0; k <= set->ninst && set->ninst > 0; ++k) {
    if (row_off) row_off[k] = set->row_off[(size_t)k];
    if (var_off) var_off[k] = set->var_off[(size_t)k];
  }
  return DP_OK;
}

int dp_matrix_info(const dp_matrix *mat, int32_t *m, int32_t *n, int64_t *nnz,
                   int64_t *padded_slots, int32_t *split_rows) {
  if (!mat) return DP_ERR_INVALID_ARG;
  if (m) *m = mat->M.m;
  if (n) *n = mat->M.n;
  if (nnz) *nnz = mat->M.nnz;
  if (padded_slots) *padded_slots = mat->padded;
  if (split_rows) *split_rows = mat->M.nsplit_rows;
  return DP_OK;
}

int dp_matrix_access_floor(dp_ctx *ctx, const dp_matrix *mat, int32_t reps, float *us) {
  dp::TraceRange trace_range("dp_matrix_access_floor");
  if (!ctx || !mat || !us || reps < 1 || mat->ctx != ctx) return DP_ERR_INVALID_ARG;
  if (mat->M.layout != dp::kLayoutEll) return DP_ERR_INVALID_ARG;
  CUDA_TRY(cudaSetDevice(ctx->device));
  cudaStream_t st = ctx->stream;
  unsigned *sink = reinterpret_cast<unsigned *>(&mat->S.ctrl->pad);  // an unused word
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) {
    if (e0) cudaEventDestroy(e0);
    cudaGetLastError();
    return DP_ERR_CUDA;
  }
  float best = -1.0f;
  int rc = DP_OK;
  for (int r = 0; r <= reps && rc == DP_OK; ++r) {  // the first launch warms up
    if (cudaEventRecord(e0, st) != cudaSuccess ||
        dp::launch_access_floor(mat->M, mat->S, sink, ctx->num_sms, st) != cudaSuccess ||
        cudaEventRecord(e1, st) != cudaSuccess || cudaEventSynchronize(e1) != cudaSuccess) {
      cudaGetLastError();
      rc = DP_ERR_CUDA;
      break;
    }
    float ms = 0.0f;
    cudaEventElapsedTime(&ms, e0, e1);
    if (r > 0 && (best < 0.0f || ms < best)) best = ms;
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (rc == DP_OK) *us = best * 1000.0f;
  return rc;
}

}  // extern "C"

namespace {

// One call's inputs on the device.
struct DevInputs {
  const double *lb, *ub, *lhs, *rhs;
  const uint8_t *vt;
};

// Device pointers are read in place, host pointers staged.
int stage_inputs(dp_ctx *ctx, dp_matrix *mat, const double *lb, const double *ub,
                 const uint8_t *vartype, const double *lhs, const double *rhs, DevInputs *d) {
  const int32_t m = mat->M.m, n = mat->M.n;
  CUDA_TRY(cudaSetDevice(ctx->device));
  cudaStream_t st = ctx->stream;
  *d = {lb, ub, lhs, rhs, vartype};
  if (n > 0) {
    if (!is_device_ptr(lb)) { CUDA_TRY(cudaMemcpyAsync(mat->st_lb, lb, 8 * (size_t)n, cudaMemcpyDefault, st)); d->lb = mat->st_lb; }
    if (!is_device_ptr(ub)) { CUDA_TRY(cudaMemcpyAsync(mat->st_ub, ub, 8 * (size_t)n, cudaMemcpyDefault, st)); d->ub = mat->st_ub; }
    if (!is_device_ptr(vartype)) { CUDA_TRY(cudaMemcpyAsync(mat->st_vt, vartype, (size_t)n, cudaMemcpyDefault, st)); d->vt = mat->st_vt; }
  }
  if (m > 0) {
    if (!is_device_ptr(lhs)) { CUDA_TRY(cudaMemcpyAsync(mat->st_lhs, lhs, 8 * (size_t)m, cudaMemcpyDefault, st)); d->lhs = mat->st_lhs; }
    if (!is_device_ptr(rhs)) { CUDA_TRY(cudaMemcpyAsync(mat->st_rhs, rhs, 8 * (size_t)m, cudaMemcpyDefault, st)); d->rhs = mat->st_rhs; }
  }
  return DP_OK;
}

// Stages inputs, writes the control block and runs the prologue.
int begin_call(dp_ctx *ctx, dp_matrix *mat, const double *lb, const double *ub,
               const uint8_t *vartype, const double *lhs, const double *rhs,
               const dp_params &p) {
  const int32_t m = mat->M.m, n = mat->M.n;
  DevInputs d;
  int rc = stage_inputs(ctx, mat, lb, ub, vartype, lhs, rhs, &d);
  if (rc) return rc;
  cudaStream_t st = ctx->stream;
  dp::Ctrl *hc = ctx->h_ctrl;
  std::memset(hc, 0, sizeof(*hc));
  hc->max_rounds = p.max_rounds;
  hc->all_active = 1;
  hc->mark_limit = mat->M.col_ptr ? n / kMarkShare : -1;
  hc->eps_int = p.eps_int;
  hc->tau_rel = p.tau_rel;
  hc->eps_feas = p.eps_feas;
  hc->inf_thr = p.inf_threshold;
  hc->wait_limit = ctx->wait_limit;
  CUDA_TRY(cudaMemcpyAsync(mat->S.ctrl, hc, sizeof(*hc), cudaMemcpyHostToDevice, st));
  CUDA_TRY(dp::launch_prologue(mat->M, mat->S, mat->vt_ws, m, n, d.lb, d.ub, d.vt, d.lhs, d.rhs,
                               p.eps_int, p.tau_rel, p.inf_threshold, ctx->num_sms, st));
  return DP_OK;
}

// Decodes the bounds into the outputs, reads the control block back and
// synchronises the stream once.
int end_call(dp_ctx *ctx, dp_matrix *mat, const dp_params &p, double *lb_out,
             double *ub_out, int32_t *infeasible, int32_t *rounds) {
  const int32_t n = mat->M.n;
  cudaStream_t st = ctx->stream;
  dp::Ctrl *hc = ctx->h_ctrl;
  if (n > 0) {
    const bool dl = is_device_ptr(lb_out), du = is_device_ptr(ub_out);
    double *o_lb = dl ? lb_out : mat->out_lb;
    double *o_ub = du ? ub_out : mat->out_ub;
    CUDA_TRY(dp::launch_epilogue(mat->S, n, o_lb, o_ub, ctx->num_sms, st));
    if (!dl) CUDA_TRY(cudaMemcpyAsync(lb_out, o_lb, 8 * (size_t)n, cudaMemcpyDefault, st));
    if (!du) CUDA_TRY(cudaMemcpyAsync(ub_out, o_ub, 8 * (size_t)n, cudaMemcpyDefault, st));
  }
  CUDA_TRY(cudaMemcpyAsync(hc, mat->S.ctrl, sizeof(*hc), cudaMemcpyDeviceToHost, st));
  CUDA_TRY(cudaStreamSynchronize(st));
  if (hc->err) return hc->err;
  *infeasible = hc->infeasible ? 1 : 0;
  *rounds = hc->round;
  if (!hc->infeasible && hc->last_changed && hc->round >= p.max_rounds && p.max_rounds > 0)
    return DP_CAP_HIT;
  return DP_OK;
}

int check_call(dp_ctx *ctx, const dp_matrix *mat, const double *lb, const double *ub,
               const uint8_t *vartype, const double *lhs, const double *rhs,
               const dp_params *params, double *lb_out, double *ub_out,
               int32_t *infeasible, int32_t *rounds, dp_params *p) {
  if (!ctx || !mat || !infeasible || !rounds) return DP_ERR_INVALID_ARG;
  if (mat->ctx != ctx) return DP_ERR_INVALID_ARG;
  const int32_t m = mat->M.m, n = mat->M.n;
  if (n > 0 && (!lb || !ub || !vartype || !lb_out || !ub_out)) return DP_ERR_INVALID_ARG;
  if (m > 0 && (!lhs || !rhs)) return DP_ERR_INVALID_ARG;
  if (params) *p = *params; else dp_params_default(p);
  if (p->max_rounds < 0 || !(p->eps_int >= 0) || !(p->tau_rel >= 0) || !(p->eps_feas >= 0) ||
      !(p->inf_threshold > 0))
    return DP_ERR_INVALID_ARG;
  return DP_OK;
}

// The whole propagation of one small problem by one team, or of every problem
// of a set by a team each; results in mat->h_res.
int team_call(dp_ctx *ctx, dp_matrix *mat, const double *lb, const double *ub,
              const uint8_t *vartype, const double *lhs, const double *rhs, const dp_params &p,
              double *lb_out, double *ub_out) {
  const size_t n = (size_t)mat->M.n;
  DevInputs d;
  int rc = stage_inputs(ctx, mat, lb, ub, vartype, lhs, rhs, &d);
  if (rc) return rc;
  cudaStream_t st = ctx->stream;
  const bool dl = n == 0 || is_device_ptr(lb_out), du = n == 0 || is_device_ptr(ub_out);
  const int32_t count = mat->ninst > 0 ? mat->ninst : 1;
  dp::TeamArgs A{};
  A.M = mat->M;
  A.rec = mat->S.rec;
  A.keys = reinterpret_cast<longlong2 *>(mat->S.keys);
  A.dirty = mat->S.dirty;
  A.mask = mat->team_mask;
  A.touch = mat->team_touch;
  A.part = mat->S.part;
  A.rowtot = mat->S.rowtot;
  A.flags = mat->team_flags;
  A.side = mat->S.side;
  A.views = mat->d_views;
  A.next = mat->team_next;
  A.lb = d.lb;
  A.ub = d.ub;
  A.lhs = d.lhs;
  A.rhs = d.rhs;
  A.vt = d.vt;
  A.lb_out = dl ? lb_out : mat->out_lb;
  A.ub_out = du ? ub_out : mat->out_ub;
  A.res = mat->h_res;
  A.count = count;
  team_params(A, p);
  const int k = team_size(
      ctx, mat->ninst > 0 ? mat->view_items : team_items(A.M.nslices, A.M.nlong), count);
  const int32_t teams = count < ctx->teams_of[k] ? count : ctx->teams_of[k];
  CUDA_TRY(dp::launch_cluster_teams(A, teams, 1 << k, ctx->num_sms, st));
  if (!dl) CUDA_TRY(cudaMemcpyAsync(lb_out, A.lb_out, 8 * n, cudaMemcpyDefault, st));
  if (!du) CUDA_TRY(cudaMemcpyAsync(ub_out, A.ub_out, 8 * n, cudaMemcpyDefault, st));
  CUDA_TRY(cudaStreamSynchronize(st));
  for (int32_t i = 0; i < count; ++i)
    if (mat->h_res[i].w) return mat->h_res[i].w;
  return DP_OK;
}

}  // namespace

extern "C" {

int dp_propagate(dp_ctx *ctx, const dp_matrix *cmat, const double *lb,
                 const double *ub, const uint8_t *vartype, const double *lhs,
                 const double *rhs, const dp_params *params, double *lb_out,
                 double *ub_out, int32_t *infeasible, int32_t *rounds) {
  dp::TraceRange trace_range("dp_propagate");
  dp_params p;
  int rc = check_call(ctx, cmat, lb, ub, vartype, lhs, rhs, params, lb_out, ub_out,
                      infeasible, rounds, &p);
  if (rc) return rc;
  dp_matrix *mat = const_cast<dp_matrix *>(cmat);
  if (mat->h_res && mat->ninst == 0 && !mat->M.val8 && mat->M.nslices <= kTeamSlices &&
      dp::single_may_be_team(ctx, mat->M.nnz)) {
    rc = team_call(ctx, mat, lb, ub, vartype, lhs, rhs, p, lb_out, ub_out);
    if (rc) return rc;
    *infeasible = mat->h_res->x;
    *rounds = mat->h_res->y;
    return mat->h_res->z ? DP_CAP_HIT : DP_OK;
  }
  rc = begin_call(ctx, mat, lb, ub, vartype, lhs, rhs, p);
  if (rc) return rc;
  if (p.max_rounds > 0) CUDA_TRY(cudaGraphLaunch(mat->exec, ctx->stream));
  return end_call(ctx, mat, p, lb_out, ub_out, infeasible, rounds);
}

int dp_propagate_persistent(dp_ctx *ctx, const dp_matrix *cmat, const double *lb,
                            const double *ub, const uint8_t *vartype, const double *lhs,
                            const double *rhs, const dp_params *params, double *lb_out,
                            double *ub_out, int32_t *infeasible, int32_t *rounds) {
  dp::TraceRange trace_range("dp_propagate_persistent");
  dp_params p;
  int rc = check_call(ctx, cmat, lb, ub, vartype, lhs, rhs, params, lb_out, ub_out,
                      infeasible, rounds, &p);
  if (rc) return rc;
  if (cmat->ninst > 0 || cmat->M.layout != dp::kLayoutEll) return DP_ERR_INVALID_ARG;
  int coop = 0;
  if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, ctx->device) != cudaSuccess ||
      !coop)
    return DP_ERR_CUDA;
  dp_matrix *mat = const_cast<dp_matrix *>(cmat);
  rc = begin_call(ctx, mat, lb, ub, vartype, lhs, rhs, p);
  if (rc) return rc;
  if (p.max_rounds > 0)
    CUDA_TRY(dp::launch_persistent(mat->M, mat->S, mat->vt_ws, ctx->num_sms, ctx->stream));
  return end_call(ctx, mat, p, lb_out, ub_out, infeasible, rounds);
}

}  // extern "C"

namespace {

// One dp_propagate_set call: the round loop as the captured graph or as one
// persistent cooperative kernel.
int set_call(dp_ctx *ctx, const dp_matrix *cset, const double *lb, const double *ub,
             const uint8_t *vartype, const double *lhs, const double *rhs,
             const dp_params *params, double *lb_out, double *ub_out, int32_t *infeasible,
             int32_t *rounds, int32_t *status, bool persistent) {
  if (!cset || cset->ninst <= 0 || !infeasible || !rounds) return DP_ERR_INVALID_ARG;
  dp_params p;
  int32_t dummy_inf = 0, dummy_rounds = 0;
  int rc = check_call(ctx, cset, lb, ub, vartype, lhs, rhs, params, lb_out, ub_out, &dummy_inf,
                      &dummy_rounds, &p);
  if (rc) return rc;
  if (persistent) {
    if (cset->M.layout != dp::kLayoutEll) return DP_ERR_INVALID_ARG;
    int coop = 0;
    if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, ctx->device) !=
            cudaSuccess ||
        !coop)
      return DP_ERR_CUDA;
  }
  dp_matrix *set = const_cast<dp_matrix *>(cset);
  if (!persistent && !set->M.val8 && set->d_views) {  // loaded for a team per problem
    rc = team_call(ctx, set, lb, ub, vartype, lhs, rhs, p, lb_out, ub_out);
    if (rc < 0) return rc;
    bool cap = false;
    for (int32_t k = 0; k < set->ninst; ++k) {
      infeasible[k] = set->h_res[k].x;
      rounds[k] = set->h_res[k].y;
      if (status) status[k] = set->h_res[k].z;
      cap |= set->h_res[k].z != 0;
    }
    return cap ? DP_CAP_HIT : DP_OK;
  }
  rc = begin_call(ctx, set, lb, ub, vartype, lhs, rhs, p);
  if (rc) return rc;
  cudaStream_t st = ctx->stream;
  const dp::InstState &I = set->S.I;
  const size_t cb = sizeof(int32_t) * (size_t)I.ninst;
  CUDA_TRY(cudaMemsetAsync(I.changed, 0, cb, st));
  CUDA_TRY(cudaMemsetAsync(I.infeasible, 0, cb, st));
  CUDA_TRY(cudaMemsetAsync(I.done, 0, cb, st));
  CUDA_TRY(cudaMemsetAsync(I.rounds, 0, cb, st));
  CUDA_TRY(cudaMemsetAsync(I.status, 0, cb, st));
  if (p.max_rounds > 0) {
    if (persistent)
      CUDA_TRY(dp::launch_persistent(set->M, set->S, set->vt_ws, ctx->num_sms, st));
    else
      CUDA_TRY(cudaGraphLaunch(set->exec, st));
  }
  int32_t *h = set->h_inst;
  CUDA_TRY(cudaMemcpyAsync(h, I.infeasible, cb, cudaMemcpyDeviceToHost, st));
  CUDA_TRY(cudaMemcpyAsync(h + I.ninst, I.rounds, cb, cudaMemcpyDeviceToHost, st));
  CUDA_TRY(cudaMemcpyAsync(h + 2 * I.ninst, I.status, cb, cudaMemcpyDeviceToHost, st));
  rc = end_call(ctx, set, p, lb_out, ub_out, &dummy_inf, &dummy_rounds);
  if (rc < 0) return rc;
  bool cap = false;
  for (int32_t k = 0; k < I.ninst; ++k) {
    infeasible[k] = h[k] ? 1 : 0;
    rounds[k] = h[I.ninst + k];
    if (status) status[k] = h[2 * I.ninst + k];
    cap |= h[2 * I.ninst + k] != 0;
  }
  return cap ? DP_CAP_HIT : DP_OK;
}

}  // namespace

extern "C" {

int dp_propagate_set(dp_ctx *ctx, const dp_matrix *cset, const double *lb, const double *ub,
                     const uint8_t *vartype, const double *lhs, const double *rhs,
                     const dp_params *params, double *lb_out, double *ub_out,
                     int32_t *infeasible, int32_t *rounds, int32_t *status) {
  dp::TraceRange trace_range("dp_propagate_set");
  return set_call(ctx, cset, lb, ub, vartype, lhs, rhs, params, lb_out, ub_out, infeasible,
                  rounds, status, false);
}

int dp_propagate_set_persistent(dp_ctx *ctx, const dp_matrix *cset, const double *lb,
                                const double *ub, const uint8_t *vartype, const double *lhs,
                                const double *rhs, const dp_params *params, double *lb_out,
                                double *ub_out, int32_t *infeasible, int32_t *rounds,
                                int32_t *status) {
  dp::TraceRange trace_range("dp_propagate_set_persistent");
  return set_call(ctx, cset, lb, ub, vartype, lhs, rhs, params, lb_out, ub_out, infeasible,
                  rounds, status, true);
}

int dp_propagate_hostloop(dp_ctx *ctx, const dp_matrix *cmat, const double *lb,
                          const double *ub, const uint8_t *vartype,
                          const double *lhs, const double *rhs,
                          const dp_params *params, double *lb_out,
                          double *ub_out, int32_t *infeasible, int32_t *rounds,
                          float *kernel_ms, int32_t *kernel_launches) {
  dp::TraceRange trace_range("dp_propagate_hostloop");
  dp_params p;
  int rc = check_call(ctx, cmat, lb, ub, vartype, lhs, rhs, params, lb_out, ub_out,
                      infeasible, rounds, &p);
  if (rc) return rc;
  dp_matrix *mat = const_cast<dp_matrix *>(cmat);
  rc = begin_call(ctx, mat, lb, ub, vartype, lhs, rhs, p);
  if (rc) return rc;
  cudaStream_t st = ctx->stream;
  const bool timed = kernel_ms != nullptr;
  constexpr int kK = 5;             // kernels of a round, in the documented order
  const int ev_of[kK] = {0, 2, 4, 8, 6};  // event pair of each (see launch_round_kernels)
  cudaEvent_t ev[10] = {};
  if (timed) {
    for (int i = 0; i < kK; ++i) kernel_ms[i] = 0.0f;
    for (int i = 0; i < 10; ++i)
      if (cudaEventCreate(&ev[i]) != cudaSuccess) {
        for (int q = 0; q < i; ++q) cudaEventDestroy(ev[q]);
        return DP_ERR_CUDA;
      }
  }
  if (kernel_launches)
    for (int i = 0; i < kK; ++i) kernel_launches[i] = 0;
  dp::Ctrl *hc = ctx->h_ctrl;
  int status = DP_OK;
  for (int32_t r = 0; r < p.max_rounds; ++r) {
    cudaError_t e = dp::launch_round_kernels(mat->M, mat->S, mat->vt_ws, 0, 0, ctx->num_sms, st,
                                             timed ? ev : nullptr);
    if (e == cudaSuccess) e = cudaMemcpyAsync(hc, mat->S.ctrl, sizeof(*hc), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) { status = DP_ERR_CUDA; break; }
    const bool split = mat->M.nsplit_rows > 0;
    const bool launched[kK] = {true, split, split, true, true};
    for (int k = 0; k < kK; ++k) {
      if (!launched[k]) continue;
      if (kernel_launches) kernel_launches[k] += 1;
      float t;
      if (timed && cudaEventElapsedTime(&t, ev[ev_of[k]], ev[ev_of[k] + 1]) == cudaSuccess)
        kernel_ms[k] += t;
    }
    if (hc->err || !hc->last_changed || hc->infeasible) break;
  }
  if (timed)
    for (int i = 0; i < 10; ++i) cudaEventDestroy(ev[i]);
  if (status) return status;
  return end_call(ctx, mat, p, lb_out, ub_out, infeasible, rounds);
}

}  // extern "C"

// ------------------------------------------------------ batched B&B nodes --

namespace dp {

bool single_may_be_team(const dp_ctx *ctx, int64_t nnz) {
  return nnz <= kTeamNnz && ctx->teams_of[0] > 0;
}

bool is_device_ptr(const void *p) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

namespace {
template <typename T>
int track_alloc(std::vector<void *> &allocs, T **p, size_t count, size_t *bytes) {
  const size_t nb = sizeof(T) * (count > 0 ? count : 1);
  if (bytes) {
    *bytes += (nb + 255) & ~(size_t)255;
    *p = nullptr;
    return DP_OK;
  }
  void *q = nullptr;
  cudaError_t e = dev_malloc(&q, nb);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return e == cudaErrorMemoryAllocation ? DP_ERR_OOM : DP_ERR_CUDA;
  }
  allocs.push_back(q);
  *p = static_cast<T *>(q);
  return DP_OK;
}

// Allocates (or, with `bytes`, only sizes) the state of a batch.
int batch_state(const DevMatrix &M, int32_t Bp, std::vector<void *> &allocs, BatchState &S,
                size_t *bytes) {
  const size_t n = (size_t)M.n, m = (size_t)M.m;
  const size_t G = (size_t)Bp / 32, Gs = (G + 3) & ~(size_t)3;
  const size_t nslots = (size_t)M.nslices * kSliceW;
  const size_t split_slots = (size_t)M.nslices_split * kSliceW;
  const size_t srows = (size_t)M.nsplit_rows;
  int rc;
#define ATRY(x) \
  if ((rc = (x)) != DP_OK) return rc
  ATRY(track_alloc(allocs, &S.cur, n * Bp, bytes));
  ATRY(track_alloc(allocs, &S.wid, n * Bp, bytes));
  ATRY(track_alloc(allocs, &S.nkey, 2 * n * Bp, bytes));
  ATRY(track_alloc(allocs, &S.chg[0], n * Gs, bytes));
  ATRY(track_alloc(allocs, &S.chg[1], n * Gs, bytes));
  ATRY(track_alloc(allocs, &S.cmask, nslots * Gs, bytes));
  ATRY(track_alloc(allocs, &S.items, G * nslots, bytes));
  ATRY(track_alloc(allocs, &S.part, split_slots * Bp, bytes));
  ATRY(track_alloc(allocs, &S.rowtot, srows * Bp, bytes));
  ATRY(track_alloc(allocs, &S.srow_act, srows * Gs, bytes));
  ATRY(track_alloc(allocs, &S.inf_bits, (size_t)kMaxGroups, bytes));
  ATRY(track_alloc(allocs, &S.chg_bits, (size_t)kMaxGroups, bytes));
  ATRY(track_alloc(allocs, &S.node_rounds, (size_t)Bp, bytes));
  ATRY(track_alloc(allocs, &S.node_status, (size_t)Bp, bytes));
  ATRY(track_alloc(allocs, &S.node_done, (size_t)Bp, bytes));
  ATRY(track_alloc(allocs, &S.alive, (size_t)kMaxGroups, bytes));
  ATRY(track_alloc(allocs, &S.fresh, (size_t)kMaxGroups, bytes));
  ATRY(track_alloc(allocs, &S.lhs, m, bytes));
  ATRY(track_alloc(allocs, &S.rhs, m, bytes));
  ATRY(track_alloc(allocs, &S.vt, n, bytes));
  ATRY(track_alloc(allocs, &S.ctrl, 1, bytes));
#undef ATRY
  S.nslots = (int64_t)nslots;
  return DP_OK;
}
}  // namespace

int alloc_batch_state(const DevMatrix &M, int32_t Bp, std::vector<void *> &allocs,
                      BatchState &S) {
  return batch_state(M, Bp, allocs, S, nullptr);
}

size_t batch_state_bytes(const DevMatrix &M, int32_t Bp) {
  std::vector<void *> none;
  BatchState S{};
  size_t bytes = 0;
  batch_state(M, Bp, none, S, &bytes);
  return bytes;
}

}  // namespace dp

namespace {

template <typename T>
int batch_alloc(BatchWs *b, T **p, size_t count) {
  void *q = nullptr;
  cudaError_t e = dp::dev_malloc(&q, sizeof(T) * (count > 0 ? count : 1));
  if (e != cudaSuccess) {
    cudaGetLastError();
    return e == cudaErrorMemoryAllocation ? DP_ERR_OOM : DP_ERR_CUDA;
  }
  b->allocs.push_back(q);
  *p = static_cast<T *>(q);
  return DP_OK;
}

// Largest node count of one launch for this matrix: a multiple of 32, at
// most 32*kMaxGroups, and small enough that entry indices (j*Bp + node,
// 32-bit) and list counts (2*n*Bp dirty entries, G*slots work items) fit in
// a signed 32-bit integer.
int32_t batch_slab(const dp_matrix *mat) {
  const int64_t n = mat->M.n > 0 ? mat->M.n : 1;
  const int64_t slots = (int64_t)mat->M.nslices * dp::kSliceW > 0
                            ? (int64_t)mat->M.nslices * dp::kSliceW : 1;
  int64_t bp = 32 * dp::kMaxGroups;
  const int64_t lim = (int64_t(1) << 30) - 1;
  while (bp >= 32 && (n * bp > lim || slots * (bp / 32) > lim)) bp -= 32;
  return (int32_t)bp;
}

// Makes (or reuses) the workspace for Bp nodes per launch.
int ensure_batch(dp_matrix *mat, int32_t Bp) {
  if (mat->batch && mat->batch->Bp_cap >= Bp) return DP_OK;
  if (mat->batch) {
    cudaStreamSynchronize(mat->ctx->stream);
    free_batch(mat->batch);
    mat->batch = nullptr;
  }
  BatchWs *b = new (std::nothrow) BatchWs();
  if (!b) return DP_ERR_OOM;
  dp::BatchState &S = b->S;
  int rc = DP_OK;
#define BTRY(x)                 \
  do {                          \
    if ((rc = (x)) != DP_OK) {  \
      free_batch(b);            \
      return rc;                \
    }                           \
  } while (0)
  BTRY(dp::alloc_batch_state(mat->M, Bp, b->allocs, S));
  if (cudaMallocHost(&b->h_ctrl, sizeof(dp::BCtrl)) != cudaSuccess ||
      cudaMallocHost(&b->h_nodes, sizeof(int32_t) * 3 * (size_t)Bp) != cudaSuccess) {
    cudaGetLastError();
    free_batch(b);
    return DP_ERR_OOM;
  }
  b->Bp_cap = Bp;
#undef BTRY
  mat->batch = b;
  return DP_OK;
}

// Makes (or reuses) the round loop of the workspace with the given activity kernel.
int ensure_batch_graph(dp_matrix *mat, dp::ActKind kind) {
  BatchWs *b = mat->batch;
  if (b->exec[kind]) return DP_OK;
  const int sms = mat->ctx->num_sms;
  const dp::DevMatrix Mc = mat->M;
  const dp::BatchState Sc = b->S;
  return build_loop_graph(
      [Mc, Sc, sms, kind](cudaGraphConditionalHandle h, cudaStream_t cs) {
        return dp::launch_batch_round(Mc, Sc, h, 1, kind, sms, cs, nullptr);
      },
      &b->graph[kind], &b->exec[kind]);
}

// Device copy of a host input (staged), or the device pointer itself.
// The staging buffer holds `cap` elements (allocated on first use).
template <typename T>
int stage_in(BatchWs *b, T **slot, const T *src, size_t count, size_t cap, cudaStream_t st,
             const T **out) {
  if (count == 0 || is_device_ptr(src)) {
    *out = src;
    return DP_OK;
  }
  if (!*slot) {
    int rc = batch_alloc(b, slot, cap);
    if (rc) return rc;
  }
  CUDA_TRY(cudaMemcpyAsync(*slot, src, sizeof(T) * count, cudaMemcpyHostToDevice, st));
  *out = *slot;
  return DP_OK;
}

constexpr int kBatchStages = 6;  // mark, mark_split, act, combine, cand_split, finish

int batch_hostloop(dp_matrix *mat, BatchWs *b, dp::ActKind kind, int32_t max_rounds, float *kernel_ms,
                   int32_t *kernel_launches) {
  dp_ctx *ctx = mat->ctx;
  cudaStream_t st = ctx->stream;
  cudaEvent_t ev[2 * kBatchStages] = {};
  const bool timed = kernel_ms != nullptr;
  if (timed)
    for (int i = 0; i < 2 * kBatchStages; ++i)
      if (cudaEventCreate(&ev[i]) != cudaSuccess) {
        for (int q = 0; q < i; ++q) cudaEventDestroy(ev[q]);
        return DP_ERR_CUDA;
      }
  const bool split = mat->M.nsplit_rows > 0;
  const bool launched[kBatchStages] = {true, split, true, split, split, true};
  int status = DP_OK;
  for (int32_t r = 0; r < max_rounds; ++r) {
    cudaError_t e = dp::launch_batch_round(mat->M, b->S, 0, 0, kind, ctx->num_sms, st,
                                           timed ? ev : nullptr);
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(b->h_ctrl, b->S.ctrl, sizeof(dp::BCtrl), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
      status = DP_ERR_CUDA;
      break;
    }
    for (int k = 0; k < kBatchStages; ++k) {
      if (!launched[k]) continue;
      if (kernel_launches) kernel_launches[k] += 1;
      float t;
      if (timed && cudaEventElapsedTime(&t, ev[2 * k], ev[2 * k + 1]) == cudaSuccess)
        kernel_ms[k] += t;
    }
    if (b->h_ctrl->err || !b->h_ctrl->any_alive) break;
  }
  if (timed)
    for (int i = 0; i < 2 * kBatchStages; ++i) cudaEventDestroy(ev[i]);
  return status;
}

// ---- nodes by teams ----

// Makes (or reuses) the state of `slots` teams over the matrix.
int ensure_teams(dp_matrix *mat, int32_t slots) {
  if (mat->teams && mat->teams->slots >= slots) return DP_OK;
  if (mat->teams) {
    cudaStreamSynchronize(mat->ctx->stream);
    free_teams(mat->teams);
    mat->teams = nullptr;
  }
  TeamWs *t = new (std::nothrow) TeamWs();
  if (!t) return DP_ERR_OOM;
  const dp::DevMatrix &M = mat->M;
  dp::TeamArgs &A = t->A;
  A.M = M;
  A.s_var = M.n;
  A.s_dirty = ((int64_t)M.n + 31) / 32;
  A.s_mask = 2 * (int64_t)M.nslices;
  A.s_touch = M.nsplit_rows;
  A.s_part = (int64_t)M.nslices_split * dp::kSliceW;
  A.side = mat->S.side;
  A.node_sums = 1;
  const size_t k = (size_t)slots;
  int rc;
#define TTRY(x)                                                         do {                                                                    if ((rc = (x)) != DP_OK) {                                              free_teams(t);                                                        return rc;                                                          }                                                                   } while (0)
  TTRY(dp::track_alloc(t->allocs, &A.rec, k * (size_t)A.s_var, nullptr));
  TTRY(dp::track_alloc(t->allocs, &A.keys, k * (size_t)A.s_var, nullptr));
  TTRY(dp::track_alloc(t->allocs, &A.dirty, k * (size_t)A.s_dirty, nullptr));
  TTRY(dp::track_alloc(t->allocs, &A.mask, k * (size_t)A.s_mask, nullptr));
  TTRY(dp::track_alloc(t->allocs, &A.touch, k * (size_t)A.s_touch, nullptr));
  TTRY(dp::track_alloc(t->allocs, &A.part, k * (size_t)A.s_part, nullptr));
  TTRY(dp::track_alloc(t->allocs, &A.rowtot, k * (size_t)A.s_touch, nullptr));
  TTRY(dp::track_alloc(t->allocs, &A.flags, k, nullptr));
  TTRY(dp::track_alloc(t->allocs, &A.next, 1, nullptr));
#undef TTRY
  if (cudaMemsetAsync(A.flags, 0, sizeof(dp::TeamFlags) * k, mat->ctx->stream) != cudaSuccess) {
    cudaGetLastError();
    free_teams(t);
    return DP_ERR_CUDA;
  }
  t->slots = slots;
  mat->teams = t;
  return DP_OK;
}

// Host bound vectors are staged kTeamStage entries at a time (more if the teams
// that run side by side hold more): a batch of many nodes over many variables and
// few nonzeros would need gigabytes else.
constexpr int64_t kTeamStage = int64_t(1) << 22;

// A device buffer for `count` staged bound vectors (the others' size grows with it).
int stage_team(TeamWs *t, double **buf, int64_t count, size_t n) {
  if (t->stage_cap < count) {
    for (double **b : {&t->st_lb, &t->st_ub, &t->out_lb, &t->out_ub}) {
      dp::dev_free(*b);
      *b = nullptr;
    }
    t->stage_cap = count;
  }
  if (*buf) return DP_OK;
  void *q = nullptr;
  const cudaError_t e =
      dp::dev_malloc(&q, sizeof(double) * (size_t)t->stage_cap * (n > 0 ? n : 1));
  if (e != cudaSuccess) {
    cudaGetLastError();
    return e == cudaErrorMemoryAllocation ? DP_ERR_OOM : DP_ERR_CUDA;
  }
  *buf = static_cast<double *>(q);
  return DP_OK;
}

// dp_propagate_nodes with a team per node.
int nodes_by_teams(dp_ctx *ctx, dp_matrix *mat, int32_t count, const double *lb, const double *ub,
                   const uint8_t *vartype, const double *lhs, const double *rhs,
                   const dp_params &p, double *lb_out, double *ub_out, int32_t *infeasible,
                   int32_t *rounds, int32_t *status) {
  const size_t n = (size_t)mat->M.n, m = (size_t)mat->M.m;
  cudaStream_t st = ctx->stream;
  const int k = team_size(ctx, team_items(mat->M.nslices, mat->M.nlong), count);
  const int32_t teams = count < ctx->teams_of[k] ? count : ctx->teams_of[k];
  int rc = ensure_teams(mat, teams);
  if (rc) return rc;
  TeamWs *t = mat->teams;
  const bool hl = n > 0 && !is_device_ptr(lb), hu = n > 0 && !is_device_ptr(ub);
  const bool hol = n > 0 && !is_device_ptr(lb_out), hou = n > 0 && !is_device_ptr(ub_out);
  int32_t per = count;  // nodes of a launch
  if (hl || hu || hol || hou)
    per = (int32_t)std::min<int64_t>(count, std::max<int64_t>(teams, kTeamStage / (int64_t)n));
  if (hl && (rc = stage_team(t, &t->st_lb, per, n))) return rc;
  if (hu && (rc = stage_team(t, &t->st_ub, per, n))) return rc;
  if (hol && (rc = stage_team(t, &t->out_lb, per, n))) return rc;
  if (hou && (rc = stage_team(t, &t->out_ub, per, n))) return rc;
  if (t->res_cap < count) {
    if (t->h_res) cudaFreeHost(t->h_res);
    t->h_res = nullptr;
    t->res_cap = 0;
    if (cudaMallocHost(&t->h_res, sizeof(int4) * (size_t)count) != cudaSuccess) {
      cudaGetLastError();
      return DP_ERR_OOM;
    }
    t->res_cap = count;
  }
  dp::TeamArgs A = t->A;
  A.vt = vartype;
  A.lhs = lhs;
  A.rhs = rhs;
  if (n > 0 && !is_device_ptr(vartype)) { CUDA_TRY(cudaMemcpyAsync(mat->st_vt, vartype, n, cudaMemcpyDefault, st)); A.vt = mat->st_vt; }
  if (m > 0 && !is_device_ptr(lhs)) { CUDA_TRY(cudaMemcpyAsync(mat->st_lhs, lhs, 8 * m, cudaMemcpyDefault, st)); A.lhs = mat->st_lhs; }
  if (m > 0 && !is_device_ptr(rhs)) { CUDA_TRY(cudaMemcpyAsync(mat->st_rhs, rhs, 8 * m, cudaMemcpyDefault, st)); A.rhs = mat->st_rhs; }
  A.in_stride = (int64_t)n;
  A.sides_ready = 1;
  team_params(A, p);
  for (int32_t s0 = 0; s0 < count; s0 += per) {
    const int32_t cnt = std::min(per, count - s0);
    const size_t off = (size_t)s0 * n, bytes = sizeof(double) * (size_t)cnt * n;
    if (hl) CUDA_TRY(cudaMemcpyAsync(t->st_lb, lb + off, bytes, cudaMemcpyDefault, st));
    if (hu) CUDA_TRY(cudaMemcpyAsync(t->st_ub, ub + off, bytes, cudaMemcpyDefault, st));
    A.lb = hl ? t->st_lb : (n > 0 ? lb + off : lb);
    A.ub = hu ? t->st_ub : (n > 0 ? ub + off : ub);
    A.lb_out = hol ? t->out_lb : (n > 0 ? lb_out + off : lb_out);
    A.ub_out = hou ? t->out_ub : (n > 0 ? ub_out + off : ub_out);
    A.res = t->h_res + s0;
    A.count = cnt;
    CUDA_TRY(dp::launch_cluster_teams(A, std::min(teams, cnt), 1 << k, ctx->num_sms, st));
    if (hol) CUDA_TRY(cudaMemcpyAsync(lb_out + off, t->out_lb, bytes, cudaMemcpyDefault, st));
    if (hou) CUDA_TRY(cudaMemcpyAsync(ub_out + off, t->out_ub, bytes, cudaMemcpyDefault, st));
  }
  CUDA_TRY(cudaStreamSynchronize(st));
  bool any_cap = false;
  for (int32_t i = 0; i < count; ++i)
    if (t->h_res[i].w) return t->h_res[i].w;
  for (int32_t i = 0; i < count; ++i) {
    const int4 r = t->h_res[i];
    infeasible[i] = r.x;
    rounds[i] = r.y;
    if (status) status[i] = r.z;
    any_cap |= r.z != 0;
  }
  return any_cap ? DP_CAP_HIT : DP_OK;
}

// Whether a team per node beats the batched kernels.
bool teams_for_nodes(const dp_ctx *ctx, const dp_matrix *mat, int32_t count) {
  if (!mat->h_res || ctx->teams_of[0] <= 0) return false;
  const int64_t nnz = mat->M.nnz, work = nnz * (int64_t)count;
  const int64_t items = team_items(mat->M.nslices, mat->M.nlong);
  // teams of one block take the nodes in several turns
  if (count > ctx->teams_of[0] && items > kTeamNodeItems) return false;
  if (mat->M.nlong == 0)
    return nnz <= kTeamNnz && work <= kTeamNodeWork &&
           items <= (int64_t)kTeamNodeShare * (kTeamWarps << team_size(ctx, items, count));
  return nnz <= kTeamNnz ? work <= kTeamNodeWork
                         : nnz <= kTeamNodeNnz && work <= kTeamNodeWorkLong;
}

// Nodes up to which a batch's chunks share warps (k_bact_few).  Measured in us
// per call (a chunk per warp / packed; random fixings and fixings at a point):
// 2.0M nonzeros with knapsack rows: 8 nodes 692 / 447 and 5350 / 3626, 16 nodes
// 755 / 601 and 5656 / 4540, 20 nodes 806 / 872 and 5828 / 6154, 32 nodes
// 855 / 923 and 5918 / 6322; 1.2M nonzeros in short rows: 16 nodes 521 / 423 and
// 3866 / 2961, 20 nodes 552 / 628 and 4017 / 4472.
constexpr int32_t kFewNodes = 16;

// Work up to which a batch without long chunks has fixed shares (k_bact<true>): its
// items times the slots of the longest.  They are even, and the ticket kernel's two
// lists and its counter cost a round 1 to 4%; above, tickets even out the memory's
// latencies.  Measured in us per call (tickets / shares): 90k nonzeros in rows of 5..7,
// 256 nodes (0.84M) 2985 / 2896; 400k, 40 nodes (0.93M) 2856 / 2759, 256 nodes (3.7M)
// 9606 / 10248; 250k in rows of 27..33, 256 nodes (2.2M) 773 / 827.
constexpr int64_t kShareWork = 1500000;

dp::ActKind act_kind(const dp::DevMatrix &M, int32_t nodes) {
  if (nodes <= kFewNodes) return dp::kActFew;
  const int64_t items = (int64_t)M.nslices * dp::kSliceW * ((nodes + 31) / 32);
  return M.max_slots < dp::kTicketSlots && M.max_slots * items <= kShareWork ? dp::kActShares
                                                                             : dp::kActTickets;
}

// How a dp_propagate_nodes call runs its rounds: the captured graph (a
// WHILE loop of the round kernels), the host (one synchronisation per round,
// so that each stage can be timed with CUDA events), or one persistent
// cooperative kernel.  The results are the same.
enum NodesMode { kNodesGraph, kNodesHostloop, kNodesPersistent };

int nodes_call(dp_ctx *ctx, const dp_matrix *cmat, int32_t count, const double *lb,
               const double *ub, const uint8_t *vartype, const double *lhs, const double *rhs,
               const dp_params *params, double *lb_out, double *ub_out, int32_t *infeasible,
               int32_t *rounds, int32_t *status, NodesMode mode, float *kernel_ms,
               int32_t *kernel_launches) {
  if (!ctx || !cmat || count < 0) return DP_ERR_INVALID_ARG;
  if (cmat->ctx != ctx || cmat->M.layout != dp::kLayoutEll) return DP_ERR_INVALID_ARG;
  if (count == 0) return DP_OK;
  if (!infeasible || !rounds) return DP_ERR_INVALID_ARG;
  dp_matrix *mat = const_cast<dp_matrix *>(cmat);
  const int32_t m = mat->M.m, n = mat->M.n;
  if (n > 0 && (!lb || !ub || !vartype || !lb_out || !ub_out)) return DP_ERR_INVALID_ARG;
  if (m > 0 && (!lhs || !rhs)) return DP_ERR_INVALID_ARG;
  dp_params p;
  if (params) p = *params; else dp_params_default(&p);
  if (p.max_rounds < 0 || !(p.eps_int >= 0) || !(p.tau_rel >= 0) || !(p.eps_feas >= 0) ||
      !(p.inf_threshold > 0))
    return DP_ERR_INVALID_ARG;
  const int32_t slab = batch_slab(mat);
  if (slab < 32) return DP_ERR_INVALID_ARG;
  CUDA_TRY(cudaSetDevice(ctx->device));
  if (mode == kNodesGraph && teams_for_nodes(ctx, mat, count))
    return nodes_by_teams(ctx, mat, count, lb, ub, vartype, lhs, rhs, p, lb_out, ub_out,
                          infeasible, rounds, status);
  cudaStream_t st = ctx->stream;
  {
    const int32_t want = count < slab ? (count + 31) / 32 * 32 : slab;
    int rc = ensure_batch(mat, want);
    if (rc) return rc;
  }
  BatchWs *b = mat->batch;
  const int32_t per = count < b->Bp_cap ? count : b->Bp_cap;
  const uint8_t *d_vt = nullptr;
  const double *d_lhs = nullptr, *d_rhs = nullptr;
  int rc;
  if ((rc = stage_in(b, &b->st_vt, vartype, (size_t)n, (size_t)n, st, &d_vt))) return rc;
  if ((rc = stage_in(b, &b->st_lhs, lhs, (size_t)m, (size_t)m, st, &d_lhs))) return rc;
  if ((rc = stage_in(b, &b->st_rhs, rhs, (size_t)m, (size_t)m, st, &d_rhs))) return rc;
  const bool host_out = n > 0 && !(is_device_ptr(lb_out) && is_device_ptr(ub_out));
  const size_t cap = (size_t)b->Bp_cap * (size_t)n;
  if (host_out && !b->out_lb) {
    if ((rc = batch_alloc(b, &b->out_lb, cap))) return rc;
    if ((rc = batch_alloc(b, &b->out_ub, cap))) return rc;
  }
  bool any_cap = false;
  for (int32_t s0 = 0; s0 < count; s0 += per) {
    dp::TraceRange batch_range("node batch launch");
    const int32_t cnt = count - s0 < per ? count - s0 : per;
    const int32_t Bp = (cnt + 31) / 32 * 32;
    const dp::ActKind kind = act_kind(mat->M, cnt);
    if (p.max_rounds > 0 && mode == kNodesGraph && (rc = ensure_batch_graph(mat, kind))) return rc;
    const size_t off = (size_t)s0 * (size_t)n, len = (size_t)cnt * (size_t)n;
    const double *d_lb = nullptr, *d_ub = nullptr;
    if ((rc = stage_in(b, &b->st_lb, n > 0 ? lb + off : lb, len, cap, st, &d_lb))) return rc;
    if ((rc = stage_in(b, &b->st_ub, n > 0 ? ub + off : ub, len, cap, st, &d_ub))) return rc;
    dp::BCtrl *hc = b->h_ctrl;
    std::memset(hc, 0, sizeof(*hc));
    hc->max_rounds = p.max_rounds;
    hc->B = cnt;
    hc->Bp = Bp;
    hc->G = Bp / 32;
    hc->any_alive = 1;
    hc->eps_int = p.eps_int;
    hc->tau_rel = p.tau_rel;
    hc->eps_feas = p.eps_feas;
    hc->inf_thr = p.inf_threshold;
    hc->wait_limit = ctx->wait_limit;
    const size_t Gs = (size_t)((Bp / 32 + 3) & ~3);
    CUDA_TRY(cudaMemcpyAsync(b->S.ctrl, hc, sizeof(*hc), cudaMemcpyHostToDevice, st));
    if (n > 0) {
      CUDA_TRY(cudaMemsetAsync(b->S.chg[0], 0, sizeof(uint32_t) * Gs * n, st));
      CUDA_TRY(cudaMemsetAsync(b->S.chg[1], 0, sizeof(uint32_t) * Gs * n, st));
    }
    CUDA_TRY(dp::launch_batch_prologue(mat->M, b->S, cnt, d_lb, d_ub, d_vt, d_lhs, d_rhs,
                                       p.eps_int, p.tau_rel, p.eps_feas, p.inf_threshold,
                                       ctx->num_sms, st));
    if (p.max_rounds > 0 && mode == kNodesGraph) CUDA_TRY(cudaGraphLaunch(b->exec[kind], st));
    if (p.max_rounds > 0 && mode == kNodesPersistent)
      CUDA_TRY(dp::launch_batch_persistent(mat->M, b->S, cnt, ctx->num_sms, st));
    if (p.max_rounds > 0 && mode == kNodesHostloop) {
      int r2 = batch_hostloop(mat, b, kind, p.max_rounds, kernel_ms, kernel_launches);
      if (r2) return r2;
    }
    if (n > 0) {
      double *o_lb = host_out ? b->out_lb : lb_out + off;
      double *o_ub = host_out ? b->out_ub : ub_out + off;
      CUDA_TRY(dp::launch_batch_epilogue(mat->M, b->S, cnt, o_lb, o_ub, ctx->num_sms, st));
      if (host_out) {
        CUDA_TRY(cudaMemcpyAsync(lb_out + off, o_lb, 8 * len, cudaMemcpyDefault, st));
        CUDA_TRY(cudaMemcpyAsync(ub_out + off, o_ub, 8 * len, cudaMemcpyDefault, st));
      }
    }
    int32_t *hn = b->h_nodes;
    CUDA_TRY(cudaMemcpyAsync(hn, b->S.inf_bits, 4 * (size_t)dp::kMaxGroups, cudaMemcpyDeviceToHost, st));
    CUDA_TRY(cudaMemcpyAsync(hn + Bp, b->S.node_rounds, 4 * (size_t)cnt, cudaMemcpyDeviceToHost, st));
    CUDA_TRY(cudaMemcpyAsync(hn + 2 * Bp, b->S.node_status, 4 * (size_t)cnt, cudaMemcpyDeviceToHost, st));
    CUDA_TRY(cudaMemcpyAsync(hc, b->S.ctrl, sizeof(*hc), cudaMemcpyDeviceToHost, st));
    CUDA_TRY(cudaStreamSynchronize(st));
    if (hc->err) return hc->err;
    for (int32_t i = 0; i < cnt; ++i) {
      infeasible[s0 + i] = (int32_t)(((uint32_t)hn[i >> 5] >> (i & 31)) & 1u);
      rounds[s0 + i] = hn[Bp + i];
      if (status) status[s0 + i] = hn[2 * Bp + i];
      any_cap |= hn[2 * Bp + i] != 0;
    }
  }
  return any_cap ? DP_CAP_HIT : DP_OK;
}

}  // namespace

extern "C" int dp_propagate_nodes(dp_ctx *ctx, const dp_matrix *mat, int32_t count,
                                  const double *lb, const double *ub, const uint8_t *vartype,
                                  const double *lhs, const double *rhs,
                                  const dp_params *params, double *lb_out, double *ub_out,
                                  int32_t *infeasible, int32_t *rounds, int32_t *status) {
  dp::TraceRange trace_range("dp_propagate_nodes");
  return nodes_call(ctx, mat, count, lb, ub, vartype, lhs, rhs, params, lb_out, ub_out,
                    infeasible, rounds, status, kNodesGraph, nullptr, nullptr);
}

extern "C" int dp_propagate_nodes_persistent(dp_ctx *ctx, const dp_matrix *mat, int32_t count,
                                             const double *lb, const double *ub,
                                             const uint8_t *vartype, const double *lhs,
                                             const double *rhs, const dp_params *params,
                                             double *lb_out, double *ub_out,
                                             int32_t *infeasible, int32_t *rounds,
                                             int32_t *status) {
  dp::TraceRange trace_range("dp_propagate_nodes_persistent");
  if (!ctx) return DP_ERR_INVALID_ARG;
  int coop = 0;
  if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, ctx->device) != cudaSuccess ||
      !coop)
    return DP_ERR_CUDA;
  return nodes_call(ctx, mat, count, lb, ub, vartype, lhs, rhs, params, lb_out, ub_out,
                    infeasible, rounds, status, kNodesPersistent, nullptr, nullptr);
}

extern "C" int dp_propagate_nodes_hostloop(dp_ctx *ctx, const dp_matrix *mat, int32_t count,
                                           const double *lb, const double *ub,
                                           const uint8_t *vartype, const double *lhs,
                                           const double *rhs, const dp_params *params,
                                           double *lb_out, double *ub_out,
                                           int32_t *infeasible, int32_t *rounds,
                                           int32_t *status, float *kernel_ms,
                                           int32_t *kernel_launches) {
  dp::TraceRange trace_range("dp_propagate_nodes_hostloop");
  if (kernel_ms)
    for (int k = 0; k < kBatchStages; ++k) kernel_ms[k] = 0.0f;
  if (kernel_launches)
    for (int k = 0; k < kBatchStages; ++k) kernel_launches[k] = 0;
  return nodes_call(ctx, mat, count, lb, ub, vartype, lhs, rhs, params, lb_out, ub_out,
                    infeasible, rounds, status, kNodesHostloop, kernel_ms, kernel_launches);
}
