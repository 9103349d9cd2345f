// Stage 3: acceptance of draft trajectories (paper Section 3.3 "Verification procedure";
// Alg. 1 Phase 1 for the high/low confidence split; Eqs. 6-7 for the top-1 fallback).
//
// One thread block per sequence.  Warps take tree nodes in turn: first the decode rule U(p) of
// every node (what threshold decoding would unmask next), then the validity of every edge, both
// as warp ballots over the block's rows; one warp then walks the tree, a lane per node.
// Integer and float compares only: the result is exact.
//
// Besides the exact and top-1 tests, the two relaxed readings of the verification test
// (the top-k-membership and probability-above-tau alternatives of that passage): membership of the drafted token in the parent's first
// topk_m candidates, and the probability of the drafted token under the parent's distribution,
// gathered here from the logits and the row's log-sum-exp (one scattered load per drafted token;
// the vocabulary pass has already produced the log-sum-exp).
//
// The joint pass of inter-block speculation (Section 3.4) verifies two trees at once: branches
// [0, n_cur) and [n_cur, B) of the same arrays.  blockIdx.y picks the tree; per-branch outputs
// keep their position in the forest, per-tree outputs are tree-major ([2, batch, ...]).
#include <algorithm>
#include "tsd_accept.cuh"

namespace tsd {

template <int WORDS>
__global__ void __launch_bounds__(kAcceptMaxThreads, 1) accept_kernel(const AcceptArgs a, const RelaxedArgs x) {
  accept_prefetch(a, blockIdx.x);
  grid_wait();
  grid_launch_next();
  const int tree = blockIdx.y;
  if (tree && a.n_branches == a.n_cur) return;  // no second tree
  accept_tree<WORDS>(a, x, blockIdx.x, tree);
}

int check_accept(const AcceptArgs& a, const RelaxedArgs& x) {
  if (a.batch < 0 || a.n_cur < 1 || a.n_cur > a.n_branches || a.n_branches < 1 || a.n_branches > kMaxBranches ||
      a.rows_per_branch < 1 || a.rows_per_branch > kMaxRows || a.top1_stride < 1)
    return TSD_ERR_INVALID_ARG;
  if (a.rule < TSD_ACCEPT_EXACT || a.rule > TSD_ACCEPT_PROB) return TSD_ERR_INVALID_ARG;
  if (a.rule == TSD_ACCEPT_TOPK && (x.topk_m < 1 || x.topk_m > a.top1_stride)) return TSD_ERR_INVALID_ARG;
  if (a.rule == TSD_ACCEPT_PROB && !x.logits) return TSD_ERR_INVALID_ARG;
  if (x.logits) {
    if (x.dtype != TSD_F32 && x.dtype != TSD_BF16) return TSD_ERR_UNSUPPORTED;
    if (!x.lse || x.vocab < 1 || x.ld < x.vocab) return TSD_ERR_INVALID_ARG;
  }
  if (a.search != TSD_SEARCH_GREEDY && a.search != TSD_SEARCH_LONGEST) return TSD_ERR_INVALID_ARG;
  if (!(a.tau == a.tau)) return TSD_ERR_INVALID_ARG;  // NaN threshold
  if (a.batch == 0) return TSD_OK;
  if (!a.parent || !a.state || !a.conf || !a.top1_idx || !a.edge_valid || !a.prefix_len || !a.accepted_node ||
      !a.accepted_len || !a.n_new_tokens || !a.unmask_flag || !a.unmask_tok)
    return TSD_ERR_INVALID_ARG;
  return TSD_OK;
}

static int launch_accept(const AcceptArgs& a, const RelaxedArgs& x) {
  if (a.batch == 0) return TSD_OK;
  const dim3 grid(a.batch, a.n_cur < a.n_branches ? 2 : 1);
  const int threads = accept_threads(std::max(a.n_cur, a.n_branches - a.n_cur));
  auto kernel = a.rows_per_branch <= 32 ? accept_kernel<1> : a.rows_per_branch <= 64 ? accept_kernel<2> : accept_kernel<kRowWords>;
  cudaError_t e = launch(kernel, grid, threads, 0, a.stream, a, x);
  return e != cudaSuccess ? cuda_fail(e, "accept_kernel") : TSD_OK;
}

int check_accept_exact(const AcceptArgs& a) {
  if (a.rule != TSD_ACCEPT_EXACT && a.rule != TSD_ACCEPT_TOP1) return TSD_ERR_INVALID_ARG;
  return check_accept(a, RelaxedArgs{});
}
int launch_accept_exact(const AcceptArgs& a) { return launch_accept(a, RelaxedArgs{}); }

}  // namespace tsd

extern "C" int tsd_accept_trajectories(int32_t batch, int32_t n_branches, int32_t rows_per_branch,
                                       const int32_t* parent, const int32_t* state, int32_t mask_id,
                                       const float* conf, const int32_t* top1_idx, int32_t top1_stride,
                                       float tau, int32_t rule, int32_t search, uint8_t* edge_valid,
                                       int32_t* prefix_len, int32_t* accepted_node,
                                       int32_t* accepted_len, int32_t* n_new_tokens,
                                       uint8_t* unmask_flag, int32_t* unmask_tok, uint32_t* status,
                                       tsd_stream_t stream) {
  return tsd_accept_joint_trees(batch, n_branches, n_branches, rows_per_branch, parent, state, mask_id, conf, top1_idx,
                                top1_stride, tau, rule, search, edge_valid, prefix_len, accepted_node, accepted_len,
                                n_new_tokens, unmask_flag, unmask_tok, status, stream);
}

extern "C" int tsd_accept_joint_trees(int32_t batch, int32_t n_branches, int32_t n_cur,
                                      int32_t rows_per_branch, const int32_t* parent, const int32_t* state,
                                      int32_t mask_id, const float* conf, const int32_t* top1_idx,
                                      int32_t top1_stride, float tau, int32_t rule, int32_t search,
                                      uint8_t* edge_valid, int32_t* prefix_len, int32_t* accepted_node,
                                      int32_t* accepted_len, int32_t* n_new_tokens, uint8_t* unmask_flag,
                                      int32_t* unmask_tok, uint32_t* status, tsd_stream_t stream) {
  const tsd::AcceptArgs a = {batch, n_branches, n_cur, rows_per_branch, parent, state, mask_id, conf, top1_idx, top1_stride,
                             tau, rule, search, edge_valid, prefix_len, accepted_node, accepted_len, n_new_tokens,
                             unmask_flag, unmask_tok, status, stream};
  const int rc = tsd::check_accept_exact(a);
  return rc != TSD_OK ? rc : tsd::launch_accept_exact(a);
}

extern "C" int tsd_accept_relaxed(int32_t batch, int32_t n_branches, int32_t n_cur, int32_t rows_per_branch,
                                  const int32_t* parent, const int32_t* state, int32_t mask_id,
                                  const float* conf, const int32_t* topk_idx, int32_t topk_stride,
                                  int32_t topk_m, const void* logits, int32_t dtype, int64_t vocab,
                                  int64_t row_stride, const float* lse, float tau, int32_t rule,
                                  int32_t search, uint8_t* edge_valid, int32_t* prefix_len,
                                  int32_t* accepted_node, int32_t* accepted_len, int32_t* n_new_tokens,
                                  uint8_t* unmask_flag, int32_t* unmask_tok, float* draft_prob,
                                  uint32_t* status, tsd_stream_t stream) {
  tsd::RelaxedArgs x{};
  x.topk_m = topk_m;
  x.logits = logits;
  x.dtype = dtype;
  x.vocab = vocab;
  x.ld = row_stride;
  x.lse = lse;
  x.draft_prob = logits ? draft_prob : nullptr;
  const tsd::AcceptArgs a = {batch, n_branches, n_cur, rows_per_branch, parent, state, mask_id, conf, topk_idx, topk_stride,
                             tau, rule, search, edge_valid, prefix_len, accepted_node, accepted_len, n_new_tokens,
                             unmask_flag, unmask_tok, status, stream};
  const int rc = tsd::check_accept(a, x);
  return rc != TSD_OK ? rc : tsd::launch_accept(a, x);
}
