// Host-side objects behind the opaque handles of the C ABI, shared by the
// library's host sources (dp_capi.cu, dp_server.cpp).
#pragma once
#include <cuda_runtime.h>
#include <cstdint>
#include <vector>

#include "dp_internal.h"

struct dp_ctx {
  int device = 0;
  int num_sms = 0;
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  dp::Ctrl *h_ctrl = nullptr;  // pinned mirror of the device control block
  int4 *h_res = nullptr;       // pinned, beside it: a single problem's team results
  int teams_of[5] = {0, 0, 0, 0, 0};  // teams of 1, 2, 4, 8, 16 blocks that fit at once
  int live_matrices = 0;
  long long wait_limit = dp::kDefaultWaitLimit;  // grid-barrier wait of the persistent loop
};

struct dp_matrix {
  dp_ctx *ctx = nullptr;
  dp::DevMatrix M{};
  dp::DevState S{};
  int64_t padded = 0;
  std::vector<void *> allocs;
  uint8_t *vt_ws = nullptr;
  // staging for host inputs / outputs
  double *st_lb = nullptr, *st_ub = nullptr, *st_lhs = nullptr, *st_rhs = nullptr;
  uint8_t *st_vt = nullptr;
  double *out_lb = nullptr, *out_ub = nullptr;
  // the round loop
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  // one team over the arrays above (dp_team.cu; sliced layout only)
  dp::TeamFlags *team_flags = nullptr;
  uint32_t *team_mask = nullptr;   // [2 * nslices]
  int32_t *team_touch = nullptr;   // [split rows]
  int4 *h_res = nullptr;           // pinned: the context's, or a set's [ninst]
  // batched nodes (allocated on the first dp_propagate_nodes call)
  struct BatchWs *batch = nullptr;
  struct TeamWs *teams = nullptr;  // few nodes of a small matrix: a team each
  const int8_t *val8 = nullptr;  // int8 copy of the values (small integers only)
  // problem sets (dp_matrix_load_set): first row / variable of each problem
  int32_t ninst = 0;
  std::vector<int32_t> row_off, var_off;
  int32_t *h_inst = nullptr;  // pinned [3*ninst], behind h_res: infeasible, rounds, status
  dp::TeamView *d_views = nullptr;  // [ninst] the problems, largest first (null: one union)
  int64_t view_items = 0;           // what the warps of the largest one's team share out
  int32_t *team_next = nullptr;
};

// State of `slots` teams (dp_team.cu) that work side by side.
struct TeamWs {
  int32_t slots = 0;
  std::vector<void *> allocs;
  dp::TeamArgs A{};             // the state's pointers and strides
  int4 *h_res = nullptr;        // pinned [res_cap]
  int32_t res_cap = 0;
  // staging of host inputs / outputs, [stage_cap] bound vectors
  double *st_lb = nullptr, *st_ub = nullptr, *out_lb = nullptr, *out_ub = nullptr;
  int64_t stage_cap = 0;
};

// Workspace of dp_propagate_nodes for up to Bp_cap nodes per launch.
struct BatchWs {
  int32_t Bp_cap = 0;
  std::vector<void *> allocs;
  dp::BatchState S{};
  dp::BCtrl *h_ctrl = nullptr;  // pinned
  int32_t *h_nodes = nullptr;   // pinned [3*Bp_cap]: infeasible, rounds, status
  // staging of host inputs / outputs, allocated when first needed
  double *st_lb = nullptr, *st_ub = nullptr, *out_lb = nullptr, *out_ub = nullptr;
  double *st_lhs = nullptr, *st_rhs = nullptr;
  uint8_t *st_vt = nullptr;
  // round loops, by dp::ActKind; each built when first needed
  cudaGraph_t graph[dp::kActKinds] = {};
  cudaGraphExec_t exec[dp::kActKinds] = {};
};

namespace dp {

// Allocates the device state of a batch of Bp nodes (a multiple of 32, at
// most 32*kMaxGroups) over matrix M; every allocation is appended to
// `allocs`, which the caller frees.  Returns DP_OK, DP_ERR_OOM or DP_ERR_CUDA.
int alloc_batch_state(const DevMatrix &M, int32_t Bp, std::vector<void *> &allocs,
                      BatchState &S);
// Device bytes alloc_batch_state takes for Bp nodes.
size_t batch_state_bytes(const DevMatrix &M, int32_t Bp);
// True for device (or managed) memory.
bool is_device_ptr(const void *p);
// Whether dp_propagate may run a problem of nnz nonzeros as one team.
bool single_may_be_team(const dp_ctx *ctx, int64_t nnz);

}  // namespace dp
