// The decode loop's own calls (Alg. 1, Sections 3.1-3.3): everything of a pass that follows the model's forward in one
// call, and the count of masked rows brought to the host without a copy.
//
// After the vocabulary pass one launch does acceptance, commit and next tree: all three belong to a sequence, so a
// block per sequence accepts with all its warps, and then one warp commits while another builds the tree.  As three
// launches they were 14 us of kernels that mostly start and wait for their first loads.
#include "tsd_accept.cuh"
#include "tsd_commit.cuh"
#include "tsd_tree.cuh"
#if defined(__x86_64__)
#include <immintrin.h>
#endif

namespace tsd {

struct AdvanceArgs {
  AcceptArgs accept;
  RelaxedArgs relaxed;
  CommitArgs commit;
  TreeArgs tree;
  uint64_t *report, *done;
  uint32_t ticket;
};

// What the host waits for: the ticket in the upper half, rows still masked and status bits below.
__device__ __forceinline__ void report_sequence(uint64_t* report, uint32_t ticket, int s, int masked, const uint32_t* status) {
  const uint32_t bits = status ? *reinterpret_cast<const volatile uint32_t*>(status) : 0u;
  *reinterpret_cast<volatile uint64_t*>(report + s) = (uint64_t)ticket << 32 | (bits & 0xffffu) << 16 | (uint32_t)masked;
}

template <int WORDS, int KK>
__global__ void __launch_bounds__(kAcceptMaxThreads, 1) advance_kernel(const __grid_constant__ AdvanceArgs a) {
  grid_wait();
  grid_launch_next();
  const int s = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int accepted = accept_tree<WORDS>(a.accept, a.relaxed, s, 0);
  __syncthreads();  // the unmask set is read below
  if (warp == 0) {
    const int masked = commit_sequence(a.commit, s, lane, accepted);
    if (a.report && lane == 0) report_sequence(a.report, a.ticket, s, masked, a.commit.status);
  } else if (warp == 1) {
    build_tree<WORDS, KK>(a.tree, s, lane, accepted);
  }
  if (a.done) {  // behind everything the block has written, for whoever sees the word: host, other streams
    __syncthreads();
    if (threadIdx.x == 0) {
      __threadfence_system();
      report_sequence(a.done, a.ticket, s, 0, nullptr);
    }
  }
}

// Start of a block: the tree is the root alone (copies in the unused slots).
__global__ void __launch_bounds__(256) begin_kernel(int B, int R, int mask_id, const int32_t* root, int32_t* parent, int32_t* state,
                                                    int32_t* n_nodes, int32_t* root_out, int32_t* fill_step, int32_t* step_base,
                                                    int32_t* n_masked, uint64_t* report, uint32_t ticket, const uint32_t* status) {
  grid_wait();
  grid_launch_next();
  const int s = blockIdx.x, t = threadIdx.x;
  bool masked = false;
  if (t < R) {
    const int32_t v = root[(size_t)s * R + t];
    masked = v == mask_id;
    root_out[(size_t)s * R + t] = v;
    fill_step[(size_t)s * R + t] = -1;
  }
  for (int i = t; i < B * R; i += blockDim.x) state[(size_t)s * B * R + i] = root[(size_t)s * R + i % R];
  for (int b = t; b < B; b += blockDim.x) parent[(size_t)s * B + b] = b == 0 ? -1 : 0;
  const int count = __syncthreads_count(masked);
  if (t == 0) {
    n_nodes[s] = 1;
    step_base[s] = 0;
    n_masked[s] = count;
    if (report) report_sequence(report, ticket, s, count, status);
  }
}

__global__ void __launch_bounds__(256) report_kernel(int batch, const int32_t* n_masked, const uint32_t* status, uint64_t* report,
                                                     uint32_t ticket) {
  grid_wait();
  grid_launch_next();
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s < batch) report_sequence(report, ticket, s, n_masked[s], status);
}

}  // namespace tsd

extern "C" int tsd_begin_block(int32_t batch, int32_t n_branches, int32_t rows_per_branch, int32_t mask_id, const int32_t* root_state,
                               int32_t* parent, int32_t* state, int32_t* n_nodes, int32_t* root_out, int32_t* fill_step,
                               int32_t* step_base, int32_t* n_masked, uint64_t* report, uint32_t ticket, const uint32_t* status,
                               tsd_stream_t stream) {
  if (batch < 0 || n_branches < 1 || n_branches > tsd::kMaxBranches || rows_per_branch < 1 || rows_per_branch > tsd::kMaxRows)
    return TSD_ERR_INVALID_ARG;
  if (batch == 0) return TSD_OK;
  if (!root_state || !parent || !state || !n_nodes || !root_out || !fill_step || !step_base || !n_masked) return TSD_ERR_INVALID_ARG;
  cudaError_t e = tsd::launch(tsd::begin_kernel, batch, 256, 0, stream, n_branches, rows_per_branch, mask_id, root_state, parent, state,
                              n_nodes, root_out, fill_step, step_base, n_masked, report, ticket, status);
  return e != cudaSuccess ? tsd::cuda_fail(e, "begin_kernel") : TSD_OK;
}

extern "C" int tsd_advance_block(const tsd_advance_args* x, tsd_stream_t stream) {
  if (!x) return TSD_ERR_INVALID_ARG;
  const int32_t S = x->batch, B = x->n_branches, R = x->rows_per_branch;
  const bool relaxed = x->rule != TSD_ACCEPT_EXACT && x->rule != TSD_ACCEPT_TOP1;
  const tsd::TopkArgs t = {x->logits, x->logits_dtype, x->n_rows, x->vocab, x->row_stride, x->k, x->conf, x->topk_idx,
                           x->topk_prob, x->lse, x->topk_workspace, x->topk_workspace_bytes, stream, tsd::kNextAfter, false};
  tsd::AdvanceArgs a = {};
  a.accept = {S, B, B, R, x->parent, x->state, x->mask_id, x->conf, x->topk_idx, x->k, x->tau, x->rule, x->search, x->edge_valid,
              x->prefix_len, x->accepted_node, x->accepted_len, x->n_new_tokens, x->unmask_flag, x->unmask_tok, x->status, stream};
  if (relaxed) a.relaxed.topk_m = x->k;
  if (x->rule == TSD_ACCEPT_PROB) {
    a.relaxed.logits = x->logits;
    a.relaxed.dtype = x->logits_dtype;
    a.relaxed.vocab = x->vocab;
    a.relaxed.ld = x->row_stride;
    a.relaxed.lse = x->lse;
    a.relaxed.draft_prob = x->draft_prob;
  }
  a.commit = {B, R, 0, x->parent, x->state, x->accepted_node, x->unmask_flag, x->unmask_tok, x->mask_id, x->tokens, x->seq_stride,
              x->block_start, x->root_out, x->fill_step, x->step_base, x->n_masked, x->status};
  a.tree = {B, R, x->k, x->state, x->accepted_node, x->unmask_flag, x->unmask_tok, x->mask_id, x->topk_idx, x->topk_prob, x->width,
            x->depth, B, B, 0, nullptr, x->next_parent, x->next_state, x->next_prob, x->next_n, x->status};
  a.report = x->report;
  a.done = x->done;
  a.ticket = x->ticket;
  int rc = tsd::check_topk(t);
  if (rc == TSD_OK) rc = tsd::check_accept(a.accept, a.relaxed);
  if (rc != TSD_OK) return rc;
  if (x->width < 1 || x->width > tsd::kTreeMaxWidth || x->depth < 0 || x->k > tsd::kTreeMaxK) return TSD_ERR_INVALID_ARG;
  const int64_t rows = (int64_t)S * B * R;  // conf, topk_* hold one each; the probability rule reads the logits of any of them
  if (x->n_rows > rows || (x->rule == TSD_ACCEPT_PROB && x->n_rows != rows)) return TSD_ERR_INVALID_ARG;
  if (x->tokens && x->seq_stride < R) return TSD_ERR_INVALID_ARG;
  if (S == 0) return TSD_OK;
  if (!x->next_parent || !x->next_state || !x->next_prob || !x->next_n || x->next_state == x->state) return TSD_ERR_INVALID_ARG;
  if ((rc = tsd::launch_topk(t)) != TSD_OK) return rc;
  const int words = (R + 31) / 32;
  auto kernel = words == 1 && x->k <= 4   ? tsd::advance_kernel<1, 4>
                : words <= 2 && x->k <= 4 ? tsd::advance_kernel<2, 4>
                                          : tsd::advance_kernel<tsd::kRowWords, tsd::kTreeMaxK>;
  cudaError_t e = tsd::launch(kernel, S, tsd::accept_threads(B), 0, stream, a);
  return e != cudaSuccess ? tsd::cuda_fail(e, "advance_kernel") : TSD_OK;
}

extern "C" int tsd_report_block(int32_t batch, const int32_t* n_masked, const uint32_t* status, uint64_t* report, uint32_t ticket,
                                tsd_stream_t stream) {
  if (batch < 1 || !n_masked || !report) return TSD_ERR_INVALID_ARG;
  cudaError_t e = tsd::launch(tsd::report_kernel, (batch + 255) / 256, 256, 0, stream, batch, n_masked, status, report, ticket);
  return e != cudaSuccess ? tsd::cuda_fail(e, "report_kernel") : TSD_OK;
}

extern "C" int tsd_wait_block(int32_t batch, const uint64_t* report, uint32_t ticket, int32_t* max_masked, uint32_t* status_bits,
                              tsd_stream_t stream) {
  if (batch < 1 || !report || !max_masked || !status_bits) return TSD_ERR_INVALID_ARG;
  const volatile uint64_t* words = report;
  int32_t most = 0;
  uint32_t bits = 0;
  bool idle = false;  // the stream had nothing left to do when it was last asked
  for (int32_t s = 0; s < batch; ++s) {
    uint64_t w;
    for (uint32_t spin = 1; (uint32_t)((w = words[s]) >> 32) != ticket; ++spin) {
#if defined(__x86_64__)
      _mm_pause();
#endif
      if (spin % 4096) continue;
      // every so often, ask whether the work this waits for can still arrive
      if (idle) return tsd::cuda_fail(cudaErrorUnknown, "tsd_wait_block: the stream is idle and has not reported this pass");
      const cudaError_t e = cudaStreamQuery(stream);
      if (e == cudaSuccess) idle = true;
      else if (e != cudaErrorNotReady) return tsd::cuda_fail(e, "tsd_wait_block");
    }
    const int32_t masked = (int32_t)(w & 0xffffu);
    most = masked > most ? masked : most;
    bits |= (uint32_t)(w >> 16) & 0xffffu;
  }
  *max_masked = most;
  *status_bits = bits;
  return TSD_OK;
}
