// Draft-tree construction (paper Alg. 1, Phase 2 "speculative expansion"; Section 3.2), the step
// right before the verification pass, fused with the root update that follows acceptance.
//
// One warp per sequence.  The next root is the accepted node's block state plus its unmask set
// (what tsd_accept_trajectories returned); the candidate pool is the top-k (token, probability) of
// every row still masked in that root, read from the scores of the pass that has just been verified
// (Section 3.1: the verification of step t provides the logits for drafting step t+1).
//   level 1  : the k most probable pool entries, one child each (root + one (row, token));
//   level > 1: every frontier node gets one child = the node + the most probable pool entry whose
//              row is still masked in it;
//   pruning  : the W most probable children of a level survive, in that order, and form the next
//              frontier; the tree stops at max_nodes nodes.
// Ties go to the lower row, then the lower rank, then the earlier child.  Lanes own rows
// (row = lane + 32 i); every selection is a warp arg-best reduction, so the result is exact and
// deterministic.  Unused node slots are copies of the root hanging off the root (an empty delta is
// never accepted).
//
// For the joint pass of inter-block speculation (Section 3.4) the tree can be written into a slice
// of a larger forest: `out_stride` branches per sequence in the output arrays, `node_base` added
// to every parent index, and a per-sequence `enable` byte (the trigger of Eq. 3) that, when 0,
// leaves the tree at its root.
#include "tsd_tree.cuh"

namespace tsd {

template <int RPL, int KK>
__global__ void __launch_bounds__(32) build_draft_tree_kernel(const TreeArgs a) {
  grid_wait();
  grid_launch_next();
  build_tree<RPL, KK>(a, blockIdx.x, threadIdx.x);
}

}  // namespace tsd

extern "C" int tsd_build_draft_tree(int32_t batch, int32_t prev_branches, int32_t rows_per_branch, int32_t k,
                                    const int32_t* prev_state, const int32_t* accepted_node,
                                    const uint8_t* unmask_flag, const int32_t* unmask_tok, int32_t mask_id,
                                    const int32_t* topk_idx, const float* topk_prob, int32_t width,
                                    int32_t depth, int32_t max_nodes, int32_t out_stride,
                                    int32_t node_base, const uint8_t* enable, int32_t* parent,
                                    int32_t* state, float* node_prob, int32_t* n_nodes, uint32_t* status,
                                    tsd_stream_t stream) {
  if (batch < 0 || prev_branches < 1 || rows_per_branch < 1 || rows_per_branch > tsd::kTreeMaxRows || k < 1 ||
      k > tsd::kTreeMaxK || width < 1 || width > tsd::kTreeMaxWidth || depth < 0 || max_nodes < 1 ||
      max_nodes > 256 || out_stride < max_nodes || node_base < 0)
    return TSD_ERR_INVALID_ARG;
  if ((unmask_flag == nullptr) != (unmask_tok == nullptr)) return TSD_ERR_INVALID_ARG;
  if (batch == 0) return TSD_OK;
  if (!prev_state || !topk_idx || !topk_prob || !parent || !state || !node_prob || !n_nodes)
    return TSD_ERR_INVALID_ARG;
  const tsd::TreeArgs a = {prev_branches, rows_per_branch, k, prev_state, accepted_node, unmask_flag, unmask_tok, mask_id,
                           topk_idx, topk_prob, width, depth, max_nodes, out_stride, node_base, enable, parent, state,
                           node_prob, n_nodes, status};
  const int rpl = (rows_per_branch + 31) / 32;
  auto kernel = rpl == 1 && k <= 4   ? tsd::build_draft_tree_kernel<1, 4>
                : rpl <= 2 && k <= 4 ? tsd::build_draft_tree_kernel<2, 4>
                                     : tsd::build_draft_tree_kernel<tsd::kTreeRowsPerLane, tsd::kTreeMaxK>;
  cudaError_t e = tsd::launch(kernel, batch, 32, 0, stream, a);
  if (e != cudaSuccess) return tsd::cuda_fail(e, "build_draft_tree_kernel");
  return TSD_OK;
}
