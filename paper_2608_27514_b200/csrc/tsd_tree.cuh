// Draft tree of one sequence's next pass, by one warp (see tsd_tree.cu).
#pragma once
#include <limits.h>
#include <math_constants.h>
#include "tsd_common.cuh"

namespace tsd {

constexpr int kTreeMaxRows = 128;   // rows per branch
constexpr int kTreeRowsPerLane = kTreeMaxRows / 32;
constexpr int kTreeMaxK = 8;
constexpr int kTreeMaxNodes = 256;
constexpr int kTreeMaxWidth = 32;   // one lane per child when a level is pruned

struct Cand {
  float p;
  int row, rank;
};
__device__ __forceinline__ bool cand_before(const Cand& a, const Cand& b) {  // a beats b
  if (b.row < 0) return a.row >= 0;
  if (a.row < 0) return false;
  if (a.p != b.p) return a.p > b.p;
  if (a.row != b.row) return a.row < b.row;
  return a.rank < b.rank;
}
// The best candidate of the warp in two warp-wide reductions (redux.sync): probabilities are
// non-negative, so their bit patterns order like unsigned integers; among the lanes that hold the
// largest one, the smallest (row, rank) wins.  Every lane returns with the winner.
__device__ __forceinline__ Cand warp_best(Cand c) {
  const unsigned full = 0xffffffffu;
  const bool valid = c.row >= 0 && c.p >= 0.f;
  const unsigned pk = valid ? (c.p > 0.f ? __float_as_uint(c.p) + 1u : 1u) : 0u;  // 0 = no candidate in this lane
  const unsigned pmax = __reduce_max_sync(full, pk);
  Cand w = {0.f, -1, 0};
  if (pmax == 0u) return w;
  const unsigned rr = (valid && pk == pmax) ? ((unsigned)c.row << 8) | (unsigned)c.rank : 0xffffffffu;
  const unsigned rmin = __reduce_min_sync(full, rr);
  w.p = __uint_as_float(pmax - 1u);  // a zero of either sign comes back as +0
  w.row = (int)(rmin >> 8);
  w.rank = (int)(rmin & 0xffu);
  return w;
}

struct TreeArgs {
  int prev_branches, R, k;
  const int32_t *prev_state, *accepted_node;
  const uint8_t* unmask_flag;
  const int32_t* unmask_tok;
  int32_t mask_id;
  const int32_t* topk_idx;
  const float* topk_prob;
  int W, D, max_nodes, out_stride, node_base;
  const uint8_t* enable;
  int32_t *parent, *state;
  float* node_prob;
  int32_t* n_nodes;
  uint32_t* status;
};

// RPL = rows per lane (R <= 32 * RPL), KK = candidates per row held in registers (k <= KK): the
// selection loops are unrolled over RPL x KK, so the common block of 32 rows with k <= 4 runs a
// tenth of the instructions of the largest case (a single warp is bound by instruction latency).
// The selection touches registers and shared memory only: a node is its parent and the (row, rank) it adds; at the end
// every node's path is written over its slot's copy of the root.  The candidates' tokens are asked for together with
// everything else, in one round trip.  `accepted`: the accepted node where the caller has it at hand (else -1 and it is loaded).
template <int RPL, int KK>
__device__ __forceinline__ void build_tree(const TreeArgs& a, int s, int lane, int accepted = -1) {
  __shared__ int s_front[kTreeMaxWidth];
  __shared__ int s_cpar[kTreeMaxWidth], s_crow[kTreeMaxWidth], s_crank[kTreeMaxWidth];
  __shared__ float s_cp[kTreeMaxWidth];
  __shared__ uint32_t s_mask[kTreeMaxNodes][RPL];  // per node: which rows are still masked
  __shared__ int s_link[kTreeMaxNodes];            // per node: parent | row << 8 | rank << 16
  __shared__ int32_t s_tok[RPL * 32][KK];          // the candidates' tokens
  const int R = a.R, k = a.k, max_nodes = a.max_nodes;
  int acc = accepted >= 0 ? accepted : a.accepted_node ? a.accepted_node[s] : 0;
  if (acc < 0 || acc >= a.prev_branches) {  // inconsistent device data: report, fall back to node 0
    if (lane == 0 && a.status) atomicOr(a.status, TSD_STATUS_BAD_PARENT);
    acc = 0;
  }
  const size_t src = ((size_t)s * a.prev_branches + acc) * R;  // rows of the accepted node
  const int32_t* idx = a.topk_idx + src * k;
  const float* prb = a.topk_prob + src * k;
  int32_t* st = a.state + (size_t)s * a.out_stride * R;
  int32_t* par = a.parent + (size_t)s * a.out_stride;
  float* np_ = a.node_prob + (size_t)s * a.out_stride;
  const int D = a.enable && !a.enable[s] ? 0 : a.D;

  // next root = accepted state + its unmask set, and the pool: this lane's rows x k, in registers
  int root[RPL];
  float pool[RPL][KK];
#pragma unroll
  for (int i = 0; i < RPL; ++i) {
    const int r = lane + 32 * i;
    root[i] = 0;
    if (r < R) {
      const int32_t old = a.prev_state[src + r];
      const bool fill = a.unmask_flag && a.unmask_flag[(size_t)s * R + r];
      const int32_t tok = a.unmask_flag ? a.unmask_tok[(size_t)s * R + r] : 0;
      root[i] = fill ? tok : old;
    }
#pragma unroll
    for (int j = 0; j < KK; ++j) pool[i][j] = (r < R && j < k) ? prb[(size_t)r * k + j] : -1.f;
#pragma unroll
    for (int j = 0; j < KK; ++j)
      if (r < R && j < k) s_tok[r][j] = idx[(size_t)r * k + j];
  }
  bool root_masked[RPL];
#pragma unroll
  for (int i = 0; i < RPL; ++i) {
    const int r = lane + 32 * i;
    root_masked[i] = r < R && root[i] == a.mask_id;
    const uint32_t word = __ballot_sync(0xffffffffu, root_masked[i]);
    if (lane == 0) s_mask[0][i] = word;
    // every node slot starts as a copy of the root
    if (r < R)
      for (int b = 0; b < max_nodes; ++b) st[(size_t)b * R + r] = root[i];
  }
  for (int b = lane; b < max_nodes; b += 32) {
    par[b] = b == 0 ? -1 : a.node_base;
    np_[b] = b == 0 ? 1.f : 0.f;
  }
  if (lane == 0) s_front[0] = 0;
  __syncwarp();

  int n = 1, n_front = 1;
  for (int level = 1; level <= D && n < max_nodes && n_front > 0; ++level) {
    int n_child = 0;
    if (level == 1) {
      // the k best pool entries: k rounds, the winner's entry is marked used in its lane
      uint32_t used = 0;
      for (int t = 0; t < k; ++t) {
        Cand best = {0.f, -1, 0};
#pragma unroll
        for (int i = 0; i < RPL; ++i) {
          const int r = lane + 32 * i;
          if (root_masked[i]) {
#pragma unroll
            for (int j = 0; j < KK; ++j) {
              if (j >= k || ((used >> (i * KK + j)) & 1u)) continue;
              const Cand c = {pool[i][j], r, j};
              if (cand_before(c, best)) best = c;
            }
          }
        }
        const Cand win = warp_best(best);
        if (win.row < 0) break;  // pool exhausted (uniform: every lane sees the same winner)
        if ((win.row & 31) == lane) used |= 1u << ((win.row >> 5) * KK + win.rank);
        if (lane == 0) { s_cpar[n_child] = 0; s_crow[n_child] = win.row; s_crank[n_child] = win.rank; s_cp[n_child] = win.p; }
        ++n_child;
      }
    } else {
      for (int f = 0; f < n_front; ++f) {
        const int node = s_front[f];
        Cand best = {0.f, -1, 0};
#pragma unroll
        for (int i = 0; i < RPL; ++i) {
          const int r = lane + 32 * i;
          if (r < R && ((s_mask[node][i] >> lane) & 1u)) {
#pragma unroll
            for (int j = 0; j < KK; ++j) {
              if (j >= k) continue;
              const Cand c = {pool[i][j], r, j};
              if (cand_before(c, best)) best = c;
            }
          }
        }
        const Cand win = warp_best(best);
        if (win.row < 0) continue;  // the node is full
        if (lane == 0) { s_cpar[n_child] = node; s_crow[n_child] = win.row; s_crank[n_child] = win.rank; s_cp[n_child] = win.p; }
        ++n_child;
      }
    }
    __syncwarp();
    // prune: lane c ranks child c by (probability descending, generation order); the first
    // min(W, budget) become nodes n, n+1, ... and the next frontier
    const int keep = min(min(a.W, max_nodes - n), n_child);
    int pos = INT_MAX;
    if (lane < n_child) {
      pos = 0;
      for (int c = 0; c < n_child; ++c)
        pos += (s_cp[c] > s_cp[lane] || (s_cp[c] == s_cp[lane] && c < lane)) ? 1 : 0;
    }
    __syncwarp();
    if (pos < keep) {
      const int node = n + pos, from = s_cpar[lane], row = s_crow[lane];
      s_front[pos] = node;
      s_link[node] = from | row << 8 | s_crank[lane] << 16;
#pragma unroll
      for (int i = 0; i < RPL; ++i) s_mask[node][i] = s_mask[from][i] & ~((row >> 5) == i ? (1u << (row & 31)) : 0u);
      par[node] = a.node_base + from;
      np_[node] = s_cp[lane];
    }
    __syncwarp();
    n += keep;
    n_front = keep;
  }
  // a lane per node: what the node and its ancestors add, over the slot's copy of the root
  for (int node = 1 + lane; node < n; node += 32) {
    for (int q = node; q > 0;) {
      const int link = s_link[q], row = (link >> 8) & 0xff, rank = link >> 16;
      st[(size_t)node * R + row] = s_tok[row][rank];
      q = link & 0xff;
    }
  }
  if (lane == 0) a.n_nodes[s] = n;
}

}  // namespace tsd
