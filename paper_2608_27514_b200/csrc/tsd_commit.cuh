// Commit of what one sequence's pass accepted, by one warp (see tsd_commit.cu).
#pragma once
#include "tsd_common.cuh"

namespace tsd {

constexpr int kCommitMaxRows = 128;
constexpr int kCommitRowsPerLane = kCommitMaxRows / 32;
constexpr int kCommitMaxBranches = 256;

struct CommitArgs {
  int B, R, root;
  const int32_t *parent, *state, *accepted_node;
  const uint8_t* unmask_flag;
  const int32_t* unmask_tok;
  int32_t mask_id;
  int32_t* tokens;
  int64_t seq_stride;
  const int32_t* block_start;
  int32_t *root_out, *fill_step, *step_base, *n_masked;
  uint32_t* status;
};

// Returns the number of rows still masked, to every lane.  `accepted`: the accepted node where the caller has it at hand
// (else -1 and it is loaded).
__device__ __forceinline__ int commit_sequence(const CommitArgs& a, int s, int lane, int accepted = -1) {
  __shared__ int s_path[kCommitMaxBranches];  // accepted node first, root last
  __shared__ int s_depth;
  const int B = a.B, R = a.R, root = a.root;
  const int32_t mask_id = a.mask_id;
  const int32_t* par = a.parent + (size_t)s * B;
  const int32_t* st = a.state + (size_t)s * B * R;
  if (lane == 0) {
    // `root` is the forest index of this tree's root (0 for a tree of its own); node and parent
    // indices are forest indices, and a tree's nodes follow its root
    int b = accepted >= 0 ? accepted : a.accepted_node ? a.accepted_node[s] : root, n = 0;
    bool bad = b < root || b >= B;
    if (bad) b = root;
    s_path[0] = b;
    while (b > root && n < B) {  // parents precede their children, so this ends within B steps
      const int p = par[b];
      if (p < root || p >= b) { bad = true; break; }
      b = p;
      s_path[++n] = b;
    }
    if (bad) {  // inconsistent tree: commit nothing but U(root)
      if (a.status) atomicOr(a.status, TSD_STATUS_BAD_PARENT);
      s_path[0] = root;
      n = 0;
    }
    s_depth = n;
  }
  __syncwarp();
  const int depth = s_depth, acc = s_path[0];
  const int base = a.step_base ? a.step_base[s] : 0;
  const int64_t start = a.block_start ? a.block_start[s] : 0;
  const bool in_range = start >= 0 && start + R <= a.seq_stride;
  if (a.tokens && !in_range && lane == 0 && a.status) atomicOr(a.status, TSD_STATUS_BAD_INDEX);
  int still = 0, open_rows = 0;
#pragma unroll
  for (int i = 0; i < kCommitRowsPerLane; ++i) {
    const int r = lane + 32 * i;
    if (r >= R) continue;
    int v = st[(size_t)acc * R + r];
    int step = -1;
    if (v == mask_id) {
      ++open_rows;
      if (a.unmask_flag && a.unmask_flag[(size_t)s * R + r]) {
        v = a.unmask_tok[(size_t)s * R + r];
        step = base + depth;
      }
    } else if (st[(size_t)root * R + r] == mask_id) {
      // filled somewhere on the path: by the shallowest node that holds it
      int j = depth;  // s_path[depth - j] is the path node at depth j
      while (j > 1 && st[(size_t)s_path[depth - j + 1] * R + r] != mask_id) --j;
      step = base + j - 1;
    }
    if (v == mask_id) ++still;
    if (a.root_out) a.root_out[(size_t)s * R + r] = v;
    if (a.tokens && in_range) a.tokens[(size_t)s * a.seq_stride + start + r] = v;
    if (a.fill_step && step >= 0) a.fill_step[(size_t)s * R + r] = step;
  }
#pragma unroll
  for (int off = 16; off; off >>= 1) {
    still += __shfl_xor_sync(0xffffffffu, still, off);
    open_rows += __shfl_xor_sync(0xffffffffu, open_rows, off);
  }
  if (lane == 0) {
    if (a.n_masked) a.n_masked[s] = still;
    if (a.step_base) a.step_base[s] = base + depth + (open_rows > 0 ? 1 : 0);
  }
  return still;
}

}  // namespace tsd
