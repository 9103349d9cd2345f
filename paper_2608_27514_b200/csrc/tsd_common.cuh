// Internal helpers shared by the tsd kernels (not part of the C ABI).
#pragma once
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>
#include "../../include/tsd.h"

namespace tsd {

// Records a failed CUDA runtime call for tsd_last_cuda_error(); returns TSD_ERR_CUDA.
int cuda_fail(cudaError_t e, const char* where);

// SMs of the GPU that the plans of the vocabulary pass and of the step were measured for.  A constant, because the workspace
// queries answer without a device; the attention, which asks for none, counts the SMs of the device it runs on.
constexpr int kPlanSms = 148;

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// ---- branch-mask blob (written by tsd_build_branch_mask, read by the attention kernels) ----
// int32 words: header[8] | cache_len[round4(S)] | records[S * n_qt], each record =
// { count, 0, (key_tile, bits) * n_kt }.  A query tile is 128 consecutive draft rows of one
// sequence = 128/R branch slots, a key tile 64 consecutive draft rows; bit (qs * 2 + w) of `bits` = slot qs of
// the query tile may read rows [32 w, 32 w + 32) of key tile `key_tile`.
constexpr int kMaskMagic = 0x54534432;
constexpr int kTile = 128;
constexpr int kKeyTile = 64;
constexpr int kHdrWords = 8;
enum { H_MAGIC = 0, H_S, H_B, H_R, H_NC, H_NQT, H_REC_WORDS, H_RECS_OFF };

struct MaskDims {
  int n_qt;        // query tiles per sequence
  int rec_words;   // words per (sequence, query tile) record
  int lens_off;    // word offset of cache_len[]
  int recs_off;    // word offset of the records
  size_t bytes;
};

inline MaskDims mask_dims(const tsd_layout& L) {
  MaskDims m;
  const int N = L.n_branches * L.rows_per_branch;
  m.n_qt = (N + kTile - 1) / kTile;
  m.rec_words = 2 + 2 * ((N + kKeyTile - 1) / kKeyTile);
  m.lens_off = kHdrWords;
  m.recs_off = kHdrWords + ((L.batch + 3) / 4) * 4;
  m.bytes = (size_t)(m.recs_off + (size_t)L.batch * m.n_qt * m.rec_words) * 4;
  m.bytes = (m.bytes + 15) / 16 * 16;
  return m;
}

int validate_layout(const tsd_layout* L);
int check_attention_args(const tsd_layout* L, const void* mask, const void* q, int64_t q_stride_b,
                         int64_t q_stride_row, int64_t q_stride_head, const void* k_cache, const void* v_cache,
                         int64_t c_stride_b, int64_t c_stride_row, int64_t c_stride_head, const void* k_draft,
                         const void* v_draft, int64_t d_stride_b, int64_t d_stride_row, int64_t d_stride_head,
                         const void* out, int64_t o_stride_b, int64_t o_stride_row, int64_t o_stride_head,
                         float sm_scale, const void* workspace);

// attention launchers (defined in their own translation units)
struct AttnArgs {
  tsd_layout L;
  const int32_t* mask;
  const void *q, *kc, *vc, *kd, *vd;
  void* out;
  float* lse;
  int64_t qs_b, qs_r, qs_h, cs_b, cs_r, cs_h, ds_b, ds_r, ds_h, os_b, os_r, os_h;
  float sm_scale;
  void* workspace;
  size_t workspace_bytes;
  uint32_t* status;
  cudaStream_t stream;
  bool concurrent;    // reads nothing that the kernel before it in the stream writes: may run beside it
  bool next_at_once;  // the next kernel may be brought up once all blocks of this one run
};
int launch_attention_simt(const AttnArgs& a);
bool attention_tc_supported(const AttnArgs& a);
size_t attention_tc_workspace_bytes(const tsd_layout& L);
int launch_attention_tc(const AttnArgs& a);
int attention_tc_blocks(const tsd_layout& L);  // that it takes, one per SM
int launch_attention(const AttnArgs& a, uint32_t flags);

// The vocabulary pass and the acceptance behind their entry points.  `launch_next`: when the next kernel may be
// brought up.  `concurrent`: the pass reads nothing that the kernel before it in the stream writes, and may run beside it.
enum { kNextAfter = 0, kNextAtTail = 1, kNextAtOnce = 2 };  // when this one is done; at the end of its rows; with its last blocks
struct TopkArgs {
  const void* logits;
  int32_t dtype;
  int64_t n_rows;
  int32_t vocab;
  int64_t row_stride;
  int32_t k;
  float* conf;
  int32_t* topk_idx;
  float *topk_prob, *lse;
  void* workspace;
  size_t workspace_bytes;
  cudaStream_t stream;
  int launch_next;
  bool concurrent;
};
int check_topk(const TopkArgs& a);
int launch_topk(const TopkArgs& a);
int64_t topk_threads(const TopkArgs& a);  // of all blocks of the pass
struct AcceptArgs {
  int32_t batch, n_branches, n_cur, rows_per_branch;
  const int32_t *parent, *state;
  int32_t mask_id;
  const float* conf;
  const int32_t* top1_idx;
  int32_t top1_stride;
  float tau;
  int32_t rule, search;
  uint8_t* edge_valid;
  int32_t *prefix_len, *accepted_node, *accepted_len, *n_new_tokens;
  uint8_t* unmask_flag;
  int32_t* unmask_tok;
  uint32_t* status;
  cudaStream_t stream;
};
int check_accept_exact(const AcceptArgs& a);  // rules EXACT and TOP1
int launch_accept_exact(const AcceptArgs& a);

// ---- programmatic dependent launch ----
// Every kernel is launched so that it may be set up while its predecessor in the stream still runs, and
// starts with grid_wait(), which holds it until that predecessor has completed and its writes are visible.
// The wait takes the pointers that are read after it, so that no load through them (read-only, hence free to
// move as far as the compiler knows) is scheduled before it.
// grid_launch_next() lets the successor's blocks be brought up from that point on; it orders nothing.  Only
// kernels of a few small blocks call it.  Where blocks fill the GPU, a successor that is placed while they
// drain piles up on the SMs that drain first: with the call in the vocabulary pass and the attention kernel,
// 416 rows of fp32 logits took 22.3 us a pass instead of 20.3 (plain launches: 22.0), an attention layer of
// 560 items 52.8 instead of 49.4 us (50.9).
// A kernel in which every block calls grid_wait() before it touches memory behaves as under a plain
// launch; what goes away is the 1-2 us of launch latency between two dependent kernels (a joint pass of six
// kernels: 131.9 -> 121.4 us; attention, vocabulary pass and acceptance of 1024 rows: 94.5 -> 89.8 us).
#ifdef __CUDACC__
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
template <typename P, typename... Q>
__device__ __forceinline__ void settle(P& pointer, Q&... more) {
  asm volatile("" : "+l"(pointer)::"memory");
  if constexpr (sizeof...(more) > 0) settle(more...);
}
template <typename... P>
__device__ __forceinline__ void grid_wait(P&... inputs) {
  grid_wait();
  settle(inputs...);
}
__device__ __forceinline__ void grid_launch_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// A kernel that may run BESIDE its predecessor A in the stream does not call grid_wait() before it reads.  What it reads was
// written before A, and A's blocks have waited for that.  Handing it on rests on
//   A: grid_wait(), grid_launch_beside() in every block   ->   this kernel's blocks start   ->   this kernel: beside_fence()
// that is, a release by all blocks of A in front of the signal that lets this kernel start, and an acquire behind the start.
// The manuals define the fences, but they name only grid_wait() as what makes memory visible across that signal:
// that a start which the signal has caused comes after it for the fences as well is an assumption of this library, and
// test_step_with_the_vocabulary_pass_beside_the_attention is what watches it (inputs rewritten in place before every step).
// The copy engine (TMA) reads through the async proxy, hence the second fence.
__device__ __forceinline__ void grid_launch_beside() {
  asm volatile("fence.acq_rel.gpu;\ngriddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void beside_fence() { asm volatile("fence.acq_rel.gpu;\nfence.proxy.async.global;" ::: "memory"); }

// `cluster`: blocks per thread-block cluster (along x).
template <typename... P, typename... A>
inline cudaError_t launch_clusters(int cluster, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                                   A... args) {
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)cluster;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}
template <typename... P, typename... A>
inline cudaError_t launch(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, A... args) {
  return launch_clusters(1, kernel, grid, block, smem, stream, args...);
}
#endif

// ---- ticket words: blocks that share a result meet without waiting for each other ----
// Each block publishes its part, then arrives on the ticket word; the last arrival reads the
// others' parts and finishes the result.  A word in use carries kTicketTag in its upper 24 bits
// and the number of arrivals so far in the lower 8; any other content counts as idle and the last
// arrival writes 0, so the memory that holds the words needs no clearing between calls.
constexpr unsigned kTicketTag = 0x7FC3A9u;

#ifdef __CUDACC__
// One arrival; true for the last of n arrivals (n <= 255).
__device__ __forceinline__ bool ticket_arrive(unsigned* t, int n) {
  unsigned old = *reinterpret_cast<volatile unsigned*>(t), assumed, cnt;
  do {
    assumed = old;
    cnt = (assumed >> 8) == kTicketTag ? (assumed & 0xffu) : 0u;
    const unsigned next = (cnt + 1 == (unsigned)n) ? 0u : ((kTicketTag << 8) | (cnt + 1));
    old = atomicCAS(t, assumed, next);
  } while (old != assumed);
  return cnt + 1 == (unsigned)n;
}
#endif

__device__ __forceinline__ float to_float(float x) { return x; }
__device__ __forceinline__ float to_float(__nv_bfloat16 x) { return __bfloat162float(x); }
__device__ __forceinline__ void from_float(float& d, float x) { d = x; }
__device__ __forceinline__ void from_float(__nv_bfloat16& d, float x) { d = __float2bfloat16_rn(x); }

}  // namespace tsd
