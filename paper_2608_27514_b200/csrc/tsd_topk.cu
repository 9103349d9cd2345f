// Stage 2: confidence and top-k candidates in one streaming pass over the logits
// (paper Eq. 2: c = max softmax(logits); Section 3.2: top-k candidates per position).
//
// HBM-bound, so the streaming loop is branch-free.  A block handles one row (or one segment of a
// row when there are few rows) in three phases:
//   1. stream: coalesced loads of 32 or 16 bytes, four 16-byte chunks per thread in flight.  Per batch the thread
//      takes the packed maximum of its 32 values, rebases its running sum to the new maximum with
//      one multiply, adds 2^(x*log2e - e) for every value (one FFMA + one ex2 each), and stores the
//      batch maximum in shared memory.
//   2. bound: the k-th largest of the warps' maxima (one shuffle reduction per warp, then every
//      warp ranks the 8 or 16 values, one per lane).  At least k values of the row are
//      >= it, so it is a valid lower bound of the k-th best.
//   3. collect: each warp re-reads only those of its batches whose maximum reaches the bound
//      (a handful per row, served by L2); the values >= bound go into a small pool in shared
//      memory, from which one warp picks the k best by counting ranks (no sort, no shuffles).
//      A pool that would overflow (heavy ties) falls back to merging per-lane lists by shuffles.
// With few rows a row is split into segments handled by different blocks.  Up to eight of them form a thread-block
// cluster and leave their partials in the shared memory of its first block; with more, the last block to finish a row
// (a ticket word in the workspace, no spinning, no clearing between calls) merges the partials.  Either way in
// segment order, so the result does not depend on arrival order.  (32 rows x 152064 in 4 segments: 9.2 us with
// tickets, 6.8 with clusters: publish, fence, ticket and re-read are a chain of global round trips.)
//
// Ordering is (logit descending, index ascending) on the raw input values (bf16 and fp32 both
// widen to fp32 exactly), so indices are uniquely defined.
#include <limits.h>
#include <math_constants.h>
#include <algorithm>
#include "tsd_common.cuh"

namespace tsd {

constexpr int kTopkUnroll = 4;            // chunks per thread per batch
constexpr int kTopkSegChunks = 32768;     // chunks per segment at most (batch maxima: 32 KB of smem)
constexpr int kTopkSmallChunks = 15360;   // chunks per row at most with 160 threads (15 KB of smem)
constexpr int kMaxSegments = 32;
constexpr int kMaxCluster = 8;            // blocks of a cluster at most (the portable size)
// How a thread's chunks lie and are read: four single ones, or two pairs of neighbours in one load each or in two.
enum { kSingle = 0, kPairs, kHalves };
constexpr int kPoolCap = 64;              // candidate pool of a block (entries)
constexpr float kLog2e = 1.4426950408889634f;

__device__ __forceinline__ bool key_before(float va, int ia, float vb, int ib) {
  return va > vb || (va == vb && ia < ib);
}

__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ uint4 ld_stream(const uint4* p) {
  uint4 r;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "l"(p));
  return r;
}

// One chunk of a pair that does not lie on 32 bytes.  Each of the pair's two loads takes half of every sector, so the second is to find
// them in L1: past L1 they are fetched twice (4096 rows of 126464 that begin 16 bytes behind a multiple of 32: 194 us, so 167-177; 200 rows
// 17.0 and 15.8).
__device__ __forceinline__ uint4 ld_half(const uint4* p) {
  uint4 r;
  asm volatile("ld.global.nc.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "l"(p));
  return r;
}

// two chunks, 32 bytes
__device__ __forceinline__ void ld_stream2(const uint4* p, uint4& a, uint4& b) {
  asm volatile("ld.global.nc.L1::no_allocate.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(a.x), "=r"(a.y), "=r"(a.z), "=r"(a.w), "=r"(b.x), "=r"(b.y), "=r"(b.z), "=r"(b.w) : "l"(p));
}

__device__ __forceinline__ void prefetch_l2(const void* p) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

// packed pairs of fp32 (one instruction for two lanes of arithmetic)
__device__ __forceinline__ uint64_t pack2(uint32_t lo, uint32_t hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(lo), "r"(hi));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& lo, float& hi) {
  uint32_t a, b;
  asm("mov.b64 {%0, %1}, %2;" : "=r"(a), "=r"(b) : "l"(v));
  lo = __uint_as_float(a);
  hi = __uint_as_float(b);
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

// Thread-block clusters: shared memory of another block, and the barrier over all threads that have not left.
__device__ __forceinline__ uint32_t cluster_address(const void* p, int rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_cluster(uint32_t a, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void cluster_arrive_relaxed() { asm volatile("barrier.cluster.arrive.relaxed;" ::: "memory"); }
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

__device__ __forceinline__ uint32_t bmax2(uint32_t a, uint32_t b) {
  uint32_t r;
  asm("max.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}

// Sorted candidate list (key order) plus the row statistics that travel with it through merges:
// the sum is kept as s * 2^e with e = fl(M * log2e) for the maximum M, so that one FFMA feeds
// the exponential; the rounding of e is undone exactly in finalize().
template <int K>
struct Acc {
  float v[K];
  int i[K];
  float e;  // exponent base; meaningful only when `seen`
  float s;
  bool seen;  // a finite value contributed

  __device__ __forceinline__ void init() {
#pragma unroll
    for (int j = 0; j < K; ++j) { v[j] = -CUDART_INF_F; i[j] = INT_MAX; }
    e = 0.f;
    s = 0.f;
    seen = false;
  }
  // insert (x, xi) if it comes before the last entry
  __device__ __forceinline__ void offer(float x, int xi) {
    if (!key_before(x, xi, v[K - 1], i[K - 1])) return;
    bool placed = false;
#pragma unroll
    for (int j = K - 1; j >= 1; --j) {
      if (!placed) {
        if (key_before(x, xi, v[j - 1], i[j - 1])) { v[j] = v[j - 1]; i[j] = i[j - 1]; }
        else { v[j] = x; i[j] = xi; placed = true; }
      }
    }
    if (!placed) { v[0] = x; i[0] = xi; }
  }
  __device__ __forceinline__ void pop_front() {
#pragma unroll
    for (int j = 0; j < K - 1; ++j) { v[j] = v[j + 1]; i[j] = i[j + 1]; }
    v[K - 1] = -CUDART_INF_F;
    i[K - 1] = INT_MAX;
  }
};

// Combines the 32 lanes' accumulators; every lane returns with the merged result.
template <int K>
__device__ __forceinline__ void warp_merge(Acc<K>& a) {
  const unsigned full = 0xffffffffu;
  float E = a.seen ? a.e : -CUDART_INF_F;
#pragma unroll
  for (int off = 16; off; off >>= 1) E = fmaxf(E, __shfl_xor_sync(full, E, off));
  float s = a.seen ? a.s * ex2_approx(a.e - E) : 0.f;
#pragma unroll
  for (int off = 16; off; off >>= 1) s += __shfl_xor_sync(full, s, off);
  float ov[K];
  int oi[K];
#pragma unroll
  for (int r = 0; r < K; ++r) {
    float bv = a.v[0];
    int bi = a.i[0];
#pragma unroll
    for (int off = 16; off; off >>= 1) {
      const float pv = __shfl_xor_sync(full, bv, off);
      const int pi = __shfl_xor_sync(full, bi, off);
      if (key_before(pv, pi, bv, bi)) { bv = pv; bi = pi; }
    }
    ov[r] = bv;
    oi[r] = bi;
    if (a.v[0] == bv && a.i[0] == bi) a.pop_front();
  }
#pragma unroll
  for (int r = 0; r < K; ++r) { a.v[r] = ov[r]; a.i[r] = oi[r]; }
  a.s = s;
  a.seen = E != -CUDART_INF_F;
  a.e = a.seen ? E : 0.f;
}

template <int K>
struct Partial {  // one segment's result, as stored in the workspace
  float e, s;     // e = -inf when nothing finite was seen
  float v[K];
  int i[K];
};

// Every lane of the warp holds the merged result; lane j writes candidate j.
template <int K>
__device__ __forceinline__ void finalize(const Acc<K>& a, int k, int64_t row, int lane, float* conf,
                                         int32_t* topk_idx, float* topk_prob, float* lse) {
  // a.s = sum 2^(x*log2e - e) with e = fl(M*log2e): the FMA residual d = M*log2e - e is exact
  const float M = a.v[0];
  const float d = fmaf(M, kLog2e, -a.e);
  const float Z = a.s * exp2f(-d);  // sum exp(x - M)
  const float inv = 1.f / Z;
#pragma unroll
  for (int j = 0; j < K; ++j) {
    if (j == lane && j < k) {
      const float p = expf(a.v[j] - M) * inv;
      topk_idx[row * k + j] = a.i[j];
      topk_prob[row * k + j] = p;
      if (j == 0) conf[row] = p;
    }
  }
  if (lse && lane == 0) lse[row] = M + logf(Z);
}

template <typename T>
struct Unpack;
template <>
struct Unpack<float> {
  static constexpr int kElems = 4;
  static constexpr uint32_t kNegInfWord = 0xff800000u;
  static __device__ __forceinline__ float chunk_max(const uint4& w) {
    return fmaxf(fmaxf(__uint_as_float(w.x), __uint_as_float(w.y)),
                 fmaxf(__uint_as_float(w.z), __uint_as_float(w.w)));
  }
  static __device__ __forceinline__ float batch_max(const uint4 (&b)[kTopkUnroll]) {
    return fmaxf(fmaxf(chunk_max(b[0]), chunk_max(b[1])), fmaxf(chunk_max(b[2]), chunk_max(b[3])));
  }
  static __device__ __forceinline__ float elem(const uint4& w, int j) {
    return __uint_as_float(j == 0 ? w.x : (j == 1 ? w.y : (j == 2 ? w.z : w.w)));
  }
  static __device__ __forceinline__ float sum_exp(const uint4& w, float ne, float s) {
    s += ex2_approx(fmaf(__uint_as_float(w.x), kLog2e, ne));
    s += ex2_approx(fmaf(__uint_as_float(w.y), kLog2e, ne));
    s += ex2_approx(fmaf(__uint_as_float(w.z), kLog2e, ne));
    s += ex2_approx(fmaf(__uint_as_float(w.w), kLog2e, ne));
    return s;
  }
};
template <>
struct Unpack<__nv_bfloat16> {
  static constexpr int kElems = 8;
  static constexpr uint32_t kNegInfWord = 0xff80ff80u;
  static __device__ __forceinline__ float batch_max(const uint4 (&b)[kTopkUnroll]) {
    uint32_t m = bmax2(bmax2(bmax2(b[0].x, b[0].y), bmax2(b[0].z, b[0].w)),
                       bmax2(bmax2(b[1].x, b[1].y), bmax2(b[1].z, b[1].w)));
    m = bmax2(m, bmax2(bmax2(bmax2(b[2].x, b[2].y), bmax2(b[2].z, b[2].w)),
                       bmax2(bmax2(b[3].x, b[3].y), bmax2(b[3].z, b[3].w))));
    return fmaxf(__uint_as_float(m << 16), __uint_as_float(m & 0xffff0000u));
  }
  static __device__ __forceinline__ float elem(const uint4& w, int j) {
    const uint32_t word = j < 2 ? w.x : (j < 4 ? w.y : (j < 6 ? w.z : w.w));
    return __uint_as_float((j & 1) ? (word & 0xffff0000u) : (word << 16));
  }
  static __device__ __forceinline__ float sum_exp(const uint4& w, float ne, float s) {
    // a bf16 pair widens to an fp32 pair with one shift and one mask; the scale-and-shift and the
    // accumulation run as packed fp32 pairs, only the exponentials are per value
    const uint64_t l2 = pack2(__float_as_uint(kLog2e), __float_as_uint(kLog2e));
    const uint64_t ne2 = pack2(__float_as_uint(ne), __float_as_uint(ne));
    uint64_t acc = pack2(0u, 0u);
    const uint32_t words[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float t0, t1;
      unpack2(fma2(pack2(words[q] << 16, words[q] & 0xffff0000u), l2, ne2), t0, t1);
      acc = add2(acc, pack2(__float_as_uint(ex2_approx(t0)), __float_as_uint(ex2_approx(t1))));
    }
    float a0, a1;
    unpack2(acc, a0, a1);
    return s + (a0 + a1);
  }
};

// grid.x = n_rows * n_seg; block = THREADS (256 when many blocks share an SM; 384 or 512 when there are so
// few rows that two or three blocks have to keep the SM busy: more warps per row; 160 where that lets all rows run at once).
template <typename T, int K, int THREADS, int LOADS>
__global__ void __launch_bounds__(THREADS)
confidence_topk_kernel(const T* __restrict__ logits, int vocab, int64_t row_stride, int k, int n_seg,
                       int chunks_per_seg, float* __restrict__ conf, int32_t* __restrict__ topk_idx,
                       float* __restrict__ topk_prob, float* __restrict__ lse,
                       Partial<K>* __restrict__ partials, unsigned* __restrict__ tickets, int prefetch, int launch_next, int rows_beside) {
  constexpr int E_ = Unpack<T>::kElems;
  constexpr int kTopkThreads = THREADS, kTopkWarps = THREADS / 32;
  constexpr int kTopkBatch = THREADS * kTopkUnroll;        // chunks per block per batch
  constexpr int kTopkMaxIter = ((THREADS == 160 ? kTopkSmallChunks : kTopkSegChunks) + kTopkBatch - 1) / kTopkBatch;  // batches per segment
  __shared__ float s_bmax[kTopkMaxIter][kTopkThreads];  // per-thread batch maxima
  __shared__ __align__(16) float s_wmax[kTopkWarps];  // per-warp maxima
  __shared__ float s_wsum[kTopkWarps];                // per-warp sums on the block's exponent base
  __shared__ float s_pool_v[kPoolCap];                // candidates found by the collect phase
  __shared__ int s_pool_i[kPoolCap];
  __shared__ int s_cnt;
  __shared__ float s_res_v[K];
  __shared__ int s_res_i[K];
  __shared__ Partial<K> s_part[kTopkWarps];           // shuffle-merge path only
  __shared__ Partial<K> s_seg[kMaxCluster];           // the segments of a row (first block of a cluster)
  const int64_t row = blockIdx.x / n_seg;
  const int seg = blockIdx.x % n_seg;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const T* rowp = logits + row * row_stride;
  const uint4* rowv = reinterpret_cast<const uint4*>(rowp);
  const int chunks_total = vocab / E_;
  const int c0 = seg * chunks_per_seg;
  const int c1 = min(c0 + chunks_per_seg, chunks_total);
  const int n_iter = (c1 - c0 + kTopkBatch - 1) / kTopkBatch;  // <= kTopkMaxIter (host-enforced)
  const bool has_tail = seg == n_seg - 1 && tid == 0 && chunks_total * E_ < vocab;
  const bool clustered = n_seg > 1 && n_seg <= kMaxCluster;
  if (rows_beside && row >= rows_beside) {
    grid_wait();
    return;
  }
  if (clustered) cluster_arrive_relaxed();  // "has started": waited for before anything is written to another block

  // Beside the kernel before it (rows_beside = rows, else 0) nothing is waited for but beside_fence() (no copy engine here).  The
  // blocks of one row more wait for that kernel, so that a kernel which waits for this one has waited for both.  (A wait by a
  // block of the last row, at its end, cost every pass 0.1 us.)
  asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %0, 0;\n@p fence.acq_rel.gpu;\n@!p griddepcontrol.wait;\n}" ::"r"(rows_beside) : "memory");
  settle(rowp, rowv);
  if (launch_next == kNextAtOnce) grid_launch_beside();

  // ---- phase 1: stream.  Two register buffers: the loads of batch it+1 are in flight while
  // batch it is processed, so a block overlaps memory latency with its own arithmetic.
  float m = -CUDART_INF_F, e = 0.f, s = 0.f;
  // Chunk u of thread t in batch `it`: single chunks, or pairs of them.  Which it is, and with it the order of the row's sum, follows from
  // the plan alone, never from an address: the same values give the same bits wherever they lie.
  auto chunk = [&](int it, int t, int u) {
    return c0 + it * kTopkBatch + (LOADS != kSingle ? 2 * t + (u & 1) + (u >> 1) * 2 * kTopkThreads : t + u * kTopkThreads);
  };
  const uint4 neg_inf = make_uint4(Unpack<T>::kNegInfWord, Unpack<T>::kNegInfWord, Unpack<T>::kNegInfWord, Unpack<T>::kNegInfWord);
  auto load_batch = [&](uint4 (&buf)[kTopkUnroll], int it) {  // past the segment: -inf adds nothing and is never a candidate
    if constexpr (LOADS == kPairs) {
#pragma unroll
      for (int u = 0; u < kTopkUnroll; u += 2) {
        const int c = chunk(it, tid, u);
        if (c + 1 < c1) {
          ld_stream2(rowv + c, buf[u], buf[u + 1]);
        } else {
          buf[u] = c < c1 ? ld_stream(rowv + c) : neg_inf;
          buf[u + 1] = neg_inf;
        }
      }
    } else {
#pragma unroll
      for (int u = 0; u < kTopkUnroll; ++u) {
        const int c = chunk(it, tid, u);
        buf[u] = c < c1 ? (LOADS == kHalves ? ld_half(rowv + c) : ld_stream(rowv + c)) : neg_inf;
      }
    }
  };
  auto process_batch = [&](const uint4 (&buf)[kTopkUnroll], int it) {
    const float bm = Unpack<T>::batch_max(buf);
    s_bmax[it][tid] = bm;
    const float m_new = fmaxf(m, bm);
    const float e_new = (m_new == -CUDART_INF_F) ? 0.f : m_new * kLog2e;
    s *= (m == -CUDART_INF_F) ? 0.f : ex2_approx(e - e_new);  // rebase: 1 when the maximum stays
    m = m_new;
    e = e_new;
    float part[kTopkUnroll];  // independent partial sums keep the dependent add chains short
    if ((it + 1) * kTopkBatch <= c1 - c0) {
#pragma unroll
      for (int u = 0; u < kTopkUnroll; ++u) part[u] = Unpack<T>::sum_exp(buf[u], -e, 0.f);
    } else {  // the segment's last, partly filled batch: no exponentials for the padding
#pragma unroll
      for (int u = 0; u < kTopkUnroll; ++u)
        part[u] = chunk(it, tid, u) < c1 ? Unpack<T>::sum_exp(buf[u], -e, 0.f) : 0.f;
    }
    s += (part[0] + part[1]) + (part[2] + part[3]);
  };
  // Optional L2 prefetch `prefetch` batches ahead of the register loads, one 128-byte line per
  // thread (the launcher turns it on for large grids only).
  auto prefetch_batch = [&](int it) {
    constexpr int kLines = kTopkBatch * 16 / 128;  // lines per batch (<= THREADS)
    const int c = c0 + it * kTopkBatch + tid * 8;  // first chunk of this thread's line
    if (tid < kLines && it < n_iter && c < c1) prefetch_l2(rowv + c);
  };
  {
    uint4 buf_a[kTopkUnroll], buf_b[kTopkUnroll];
    if (n_iter > 0) load_batch(buf_a, 0);
    for (int p = 1; p <= prefetch; ++p) prefetch_batch(p);
    for (int it = 0; it < n_iter; it += 2) {
      if (it + 1 < n_iter) load_batch(buf_b, it + 1);
      if (prefetch) { prefetch_batch(it + prefetch + 1); prefetch_batch(it + prefetch + 2); }
      process_batch(buf_a, it);
      if (it + 1 < n_iter) {
        if (it + 2 < n_iter) load_batch(buf_a, it + 2);
        process_batch(buf_b, it + 1);
      }
    }
  }
  float tail_max = -CUDART_INF_F;
  if (has_tail) {  // ragged tail of a vocabulary that is not a multiple of the chunk size
    for (int x = chunks_total * E_; x < vocab; ++x) tail_max = fmaxf(tail_max, to_float(rowp[x]));
    const float m_new = fmaxf(m, tail_max);
    const float e_new = (m_new == -CUDART_INF_F) ? 0.f : m_new * kLog2e;
    s *= (m == -CUDART_INF_F) ? 0.f : ex2_approx(e - e_new);
    m = m_new;
    e = e_new;
    for (int x = chunks_total * E_; x < vocab; ++x) s += ex2_approx(fmaf(to_float(rowp[x]), kLog2e, -e));
  }

  if (launch_next == kNextAtTail) grid_launch_next();

  // ---- phase 2: bound = k-th largest of the warps' maxima.  Each of the k best warps holds a
  // value equal to its maximum, so at least k values of the segment reach the bound.  One shuffle
  // reduction per warp, one block-wide barrier, then a rank count per warp.
  if (tid == 0) s_cnt = 0;
  {
    float wm = m;
#pragma unroll
    for (int off = 16; off; off >>= 1) wm = fmaxf(wm, __shfl_xor_sync(0xffffffffu, wm, off));
    if (lane == 0) s_wmax[warp] = wm;
  }
  __syncthreads();
  // lane l < WARPS takes warp maximum l and counts the maxima that come before it (larger, or
  // equal from a lower warp): ranks are unique, rank 0 is the block maximum, rank K-1 the bound
  float M, bound;
  {
    const float mine = lane < kTopkWarps ? s_wmax[lane] : -CUDART_INF_F;
    int rank = 0;
#pragma unroll
    for (int q = 0; q < kTopkWarps; ++q) {
      const float o = s_wmax[q];
      rank += (o > mine || (o == mine && q < lane)) ? 1 : 0;
    }
    const bool in = lane < kTopkWarps;
    const unsigned b0 = __ballot_sync(0xffffffffu, in && rank == 0);
    const unsigned bk = __ballot_sync(0xffffffffu, in && rank == K - 1);
    M = __shfl_sync(0xffffffffu, mine, __ffs(b0) - 1);
    bound = __shfl_sync(0xffffffffu, mine, __ffs(bk) - 1);
  }
  // the block's sum on the block's exponent base; the per-warp sums meet after the next barrier
  const float E = (M == -CUDART_INF_F) ? 0.f : M * kLog2e;
  {
    float sr = (m == -CUDART_INF_F) ? 0.f : s * ex2_approx(e - E);
#pragma unroll
    for (int off = 16; off; off >>= 1) sr += __shfl_xor_sync(0xffffffffu, sr, off);
    if (lane == 0) s_wsum[warp] = sr;
  }

  // ---- phase 3: collect the values >= bound from the few batches that hold one
  Acc<K> a;
  a.init();
  // The whole block waits for its slowest warp here, so a hit batch (32 values for bf16, 16 for
  // fp32) is examined by the warp together: lane l re-reads value l of the batch (an L2 hit) and
  // offers it to its own list.
  for (int it = 0; it < n_iter; ++it) {
    unsigned hits = __ballot_sync(0xffffffffu, s_bmax[it][tid] >= bound);
    while (hits) {
      const int src = __ffs(hits) - 1;
      hits &= hits - 1;
      if (lane < kTopkUnroll * E_) {
        const int c = chunk(it, warp * 32 + src, lane / E_);
        if (c < c1) {
          const int xi = c * E_ + lane % E_;
          const float x = to_float(rowp[xi]);
          if (x >= bound) a.offer(x, xi);
        }
      }
    }
  }
  if (has_tail && tail_max >= bound) {
    for (int x = chunks_total * E_; x < vocab; ++x) {
      const float v = to_float(rowp[x]);
      if (v >= bound) a.offer(v, x);
    }
  }
  // The lanes that found something (a handful per block) put their entries into a small pool in
  // shared memory.  If the pool would overflow (heavy ties: many values equal to the bound), the
  // lists are merged by shuffles instead, which is slower but has no capacity.
  {
    int n_mine = 0;
#pragma unroll
    for (int j = 0; j < K; ++j) n_mine += a.i[j] != INT_MAX;
    if (n_mine > 0) {
      const int at = atomicAdd(&s_cnt, n_mine);
      if (at + n_mine <= kPoolCap) {
#pragma unroll
        for (int j = 0; j < K; ++j)
          if (j < n_mine) { s_pool_v[at + j] = a.v[j]; s_pool_i[at + j] = a.i[j]; }
      }
    }
  }
  __syncthreads();
  const int n_pool = s_cnt;
  if (n_pool > kPoolCap) {
    a.seen = m != -CUDART_INF_F;
    a.e = e;
    a.s = s;
    warp_merge(a);
    if (lane == 0) {
      s_part[warp].e = a.seen ? a.e : -CUDART_INF_F;
      s_part[warp].s = a.s;
#pragma unroll
      for (int j = 0; j < K; ++j) { s_part[warp].v[j] = a.v[j]; s_part[warp].i[j] = a.i[j]; }
    }
    __syncthreads();
    if (warp != 0) return;
    a.init();
    if (lane < kTopkWarps) {
      a.seen = s_part[lane].e != -CUDART_INF_F;
      a.e = a.seen ? s_part[lane].e : 0.f;
      a.s = s_part[lane].s;
#pragma unroll
      for (int j = 0; j < K; ++j) { a.v[j] = s_part[lane].v[j]; a.i[j] = s_part[lane].i[j]; }
    }
    warp_merge(a);
  } else {
    if (warp != 0) return;
    // sum of the warps' sums (fixed tree), and the pool's best K by rank: every lane counts the
    // entries that come before its own (keys are unique), so rank r goes to slot r without a sort
    float st = lane < kTopkWarps ? s_wsum[lane] : 0.f;
#pragma unroll
    for (int off = 16; off; off >>= 1) st += __shfl_xor_sync(0xffffffffu, st, off);
    if (lane < K) { s_res_v[lane] = -CUDART_INF_F; s_res_i[lane] = INT_MAX; }
    __syncwarp();
#pragma unroll
    for (int h = 0; h < kPoolCap / 32; ++h) {
      const int q = lane + 32 * h;
      if (q < n_pool) {
        const float v = s_pool_v[q];
        const int i = s_pool_i[q];
        int rank = 0;
        for (int o = 0; o < n_pool; ++o) rank += key_before(s_pool_v[o], s_pool_i[o], v, i);
        if (rank < K) { s_res_v[rank] = v; s_res_i[rank] = i; }
      }
    }
    __syncwarp();
#pragma unroll
    for (int j = 0; j < K; ++j) { a.v[j] = s_res_v[j]; a.i[j] = s_res_i[j]; }
    a.seen = M != -CUDART_INF_F;
    a.e = E;
    a.s = st;
  }
  if (n_seg == 1) {
    finalize(a, k, row, lane, conf, topk_idx, topk_prob, lse);
    return;
  }
  if (clustered) {
    cluster_wait();
    const uint32_t to = cluster_address(&s_seg[seg], 0);
    if (lane == 0) {
      st_cluster(to, a.seen ? a.e : -CUDART_INF_F);
      st_cluster(to + 4, a.s);
    }
#pragma unroll
    for (int j = 0; j < K; ++j)
      if (lane == j) {
        st_cluster(to + 8 + 4 * j, a.v[j]);
        st_cluster(to + 8 + 4 * K + 4 * j, __int_as_float(a.i[j]));
      }
    cluster_arrive();
    if (seg != 0) return;
    cluster_wait();
    a.init();
    if (lane < n_seg) {
      const float pe = s_seg[lane].e;
      a.seen = pe != -CUDART_INF_F;
      a.e = a.seen ? pe : 0.f;
      a.s = s_seg[lane].s;
#pragma unroll
      for (int j = 0; j < K; ++j) { a.v[j] = s_seg[lane].v[j]; a.i[j] = s_seg[lane].i[j]; }
    }
    warp_merge(a);
    finalize(a, k, row, lane, conf, topk_idx, topk_prob, lse);
    return;
  }
  // many segments per row: publish this one, the last to arrive merges all of them
  bool last = false;
  if (lane == 0) {
    Partial<K>* p = partials + row * n_seg + seg;
    p->e = a.seen ? a.e : -CUDART_INF_F;
    p->s = a.s;
#pragma unroll
    for (int j = 0; j < K; ++j) { p->v[j] = a.v[j]; p->i[j] = a.i[j]; }
    __threadfence();
    last = ticket_arrive(tickets + row, n_seg);
    __threadfence();
  }
  if (!__shfl_sync(0xffffffffu, last, 0)) return;
  a.init();
  if (lane < n_seg) {
    const Partial<K>* p = partials + row * n_seg + lane;
    const float pe = __ldcg(&p->e);
    a.seen = pe != -CUDART_INF_F;
    a.e = a.seen ? pe : 0.f;
    a.s = __ldcg(&p->s);
#pragma unroll
    for (int j = 0; j < K; ++j) { a.v[j] = __ldcg(&p->v[j]); a.i[j] = __ldcg(&p->i[j]); }
  }
  warp_merge(a);
  finalize(a, k, row, lane, conf, topk_idx, topk_prob, lse);
}

struct TopkPlan {
  int n_seg, chunks_per_seg, K, threads, prefetch;
  size_t partial_bytes, ticket_off, total_bytes;
};

static int round_k(int k) { return k <= 4 ? k : (k <= 6 ? 6 : 8); }

static void scratch_layout(int64_t n_rows, TopkPlan& p) {
  const size_t rec = 8 + 8 * (size_t)p.K;
  p.partial_bytes = (size_t)n_rows * p.n_seg * rec;
  p.ticket_off = (p.partial_bytes + 15) / 16 * 16;
  p.total_bytes = p.n_seg > 1 ? p.ticket_off + ((size_t)n_rows * 4 + 15) / 16 * 16 : 0;
}

// The workspace query's answer: room for as many segments as give every SM at least one block, whether or not a
// plan uses as many, so that the size a caller has to provide does not follow the tuning of the plans.
static size_t workspace_bytes(int64_t n_rows, int vocab, int k, int elems_per_chunk) {
  const int chunks = vocab / elems_per_chunk;
  TopkPlan p;
  p.K = round_k(k);
  const int64_t n_seg = std::min<int64_t>(std::min<int64_t>((kPlanSms + n_rows - 1) / n_rows, kMaxSegments), std::max(1, chunks / 2048));
  p.n_seg = (int)std::max<int64_t>(n_seg, (chunks + kTopkSegChunks - 1) / kTopkSegChunks);
  scratch_layout(n_rows, p);
  return p.total_bytes;
}

static TopkPlan topk_plan(int64_t n_rows, int vocab, int k, int elems_per_chunk) {
  TopkPlan p;
  p.K = round_k(k);
  const int chunks = vocab / elems_per_chunk;
  // Few rows are split into 2, 4 or 8 segments where that shortens what the busiest SM streams, in rows of 126464 bf16
  // (7.3 us each), by more than a split costs (1.2 us and a little per segment).  Measured, 126464 bf16: 8 rows whole
  // 9.1 us, in 8 segments 5.7; 50 rows 11.0, in 2 9.1, in 8 8.6; 74 rows 11.2, in 2 9.8, in 4 10.4; 100 rows 11.6, in 4
  // 11.2; 148 rows 12.3, in 2 12.7; 200 rows 16.7, in 2 15.8; 256 rows 17.1, in 2 18.1; of 32000: 32 rows 5.0, in 4 5.5.
  int64_t n_seg = 1;
  if (n_rows > 0 && n_rows <= 222) {
    double best = 1e30;
    for (int n = 1; n <= (n_rows <= kPlanSms ? kMaxCluster : 2); n *= 2) {
      const double rounds = (double)((n_rows * n + kPlanSms - 1) / kPlanSms) / n;
      const double cost = rounds * chunks / 15808 + (n > 1 ? 0.17 + 0.005 * n : 0.0);
      if (cost < best) { best = cost; n_seg = n; }
    }
  }
  // a segment may span at most kTopkSegChunks chunks (its batch maxima live in shared memory)
  n_seg = std::max<int64_t>(n_seg, (chunks + kTopkSegChunks - 1) / kTopkSegChunks);
  p.n_seg = (int)std::max<int64_t>(n_seg, 1);
  // As many warps per row as still give every block a slot at once: 256 x 126464 bf16 with 512 threads 17.0 us, with
  // 384 17.9, with 256 18.8; 444 x 126464 25.0 / 23.5 / 24.4; 960 x 126464 50.2 / 48.2 / 46.0.
  const int64_t units = n_rows * p.n_seg;
  p.threads = units <= 2 * kPlanSms ? 512 : (units <= 3 * kPlanSms ? 384 : 256);
  // Long rows, a few more than 256 threads per row leave room for at one time, would be finished by a second wave of few blocks.
  // fp32: 160 threads, of which 7 blocks run per SM, up to 1036 rows (of 50257, with 256 threads and with 160: 800 rows 37.0 and 30.7 us, 1024 rows
  // 42.7 and 37.2, 1100 rows 43.8 and 47.2; of 32000: 800 rows 24.2 and 22.3).  bf16: 384, whose two waves are more even (of 126464, with
  // 256 and 384: 640 rows 37.1 and 35.6, 740 rows 40.7 and 36.7, 800 rows 41.6 and 42.2; of 152064: 740 rows 45.8 and 41.4).
  if (elems_per_chunk == 4 && units > 5 * kPlanSms && units <= 7 * kPlanSms && p.K <= 4 && chunks > 4096 && chunks <= kTopkSmallChunks) p.threads = 160;
  if (elems_per_chunk == 8 && units > 4 * kPlanSms && units <= 5 * kPlanSms && chunks > 8192) p.threads = 384;
  // Rows that even 256 threads walk in one batch: with 512 threads 256 x 4096 fp32 takes 4.6 us and with 256 4.3, bf16 4.7 and 4.4,
  // 256 x 8192 bf16 4.8 and 4.6, 296 x 8000 bf16 5.2 and 4.9; 128 x 8000 and fewer rows the same (4.3).  128 x 16000: 5.0 and 5.8.
  if (chunks <= 1024) p.threads = 256;
  // clusters of large blocks are hard to place: 74 x 126464 in 4 segments 12.8 us with 512 threads, 10.4 with 256
  if (p.n_seg > 1 && units > kPlanSms) p.threads = 256;
  // L2 prefetch distance in batches (measured): with very many waves of blocks, requesting lines three batches ahead
  // adds 2 % of bandwidth (16384 x 126464: 687 us, without 700); with fewer it delays the demand loads (4096 x 32000:
  // 57.0 us, without 53.6; 4096 x 126464: 171 and 167; 4096 x 152064: 189.7 and 190.8)
  p.prefetch = units >= 8192 ? 3 : 0;
  p.chunks_per_seg = (chunks + p.n_seg - 1) / p.n_seg;
  if (p.n_seg > 1) p.chunks_per_seg += p.chunks_per_seg & 1;
  if (p.chunks_per_seg == 0) p.chunks_per_seg = 1;
  scratch_layout(n_rows, p);
  if (p.n_seg <= kMaxCluster) p.total_bytes = 0;  // the segments meet in shared memory
  return p;
}

template <typename T, int K>
static auto pick_kernel(int threads, int loads) {
  auto kernel = threads == 512 ? confidence_topk_kernel<T, K, 512, kSingle>
              : threads == 384 ? confidence_topk_kernel<T, K, 384, kSingle> : confidence_topk_kernel<T, K, 256, kSingle>;
  // (a block ranks its warps' maxima: it needs as many warps as candidates)
  if constexpr (K <= 4 && sizeof(T) == 4)
    if (threads == 160) kernel = confidence_topk_kernel<T, K, 160, kSingle>;
  if constexpr (sizeof(T) == 2) {  // (rows in segments get 512 or 256 threads, 2048 rows and more 256)
    if (loads == kPairs) kernel = threads == 512 ? confidence_topk_kernel<T, K, 512, kPairs> : confidence_topk_kernel<T, K, 256, kPairs>;
    if (loads == kHalves) kernel = threads == 512 ? confidence_topk_kernel<T, K, 512, kHalves> : confidence_topk_kernel<T, K, 256, kHalves>;
  }
  return kernel;
}

template <typename T, int K>
static cudaError_t run_plan(const TopkArgs& a, const TopkPlan& p, void* ws) {
  Partial<K>* partials = reinterpret_cast<Partial<K>*>(ws);
  unsigned* tickets = reinterpret_cast<unsigned*>(static_cast<char*>(ws) + p.ticket_off);
  // bf16: chunks in pairs, read 32 bytes at a time where every row (and, as segments are of whole pairs, every segment) begins on 32 bytes.
  // For rows in segments and for many rows: with 16- and 32-byte loads, 32 rows of 152064 6.25 and 5.93 us, 128 rows of 126464 12.2 and 11.6, 16384
  // rows 648 and 626.  In between the pass alone gains too (320 rows 22.9 and 22.5, 1024 rows 47.0 and 46.3), but behind an attention
  // kernel it loses (16 us of attention and 320 rows: 39.5 and 40.3; a joint pass of 1280 rows 110.4 and 111.2); the cause has not been found.
  // Rows in segments gain there (steps of 152064, single chunks and pairs: 96 rows and 96 items 26.1 and 25.6 us, 160 and 160 40.4 and 39.3, 192 and
  // 192 41.6 and 40.5), except where a few run beside a short attention (32 items of 12 tiles: 32 rows 16.0 and 16.5, 64 rows 17.4 and 17.55).
  // The rule does not look at the position, because a step has to give the bits of its single calls.
  // fp32 has half the arithmetic per byte and gains nothing (416 x 50257: 18.3 and 19.1).
  // Segments too short to give most threads a pair keep single chunks (8 segments under 512 threads, single and in pairs: 8 rows of 32000, 500
  // chunks per segment, 5.10 and 5.37 us; of 36000, 564 chunks, 5.19 and 5.33; of 40000, 626, 5.27 and 5.30; 18 rows of 48000, 750, 5.71 and 5.54).
  int loads = kSingle;
  if (sizeof(T) == 2 && (p.n_seg > 1 ? 4 * p.chunks_per_seg > 5 * p.threads : a.n_rows >= 2048))
    loads = a.row_stride % 16 == 0 && reinterpret_cast<uintptr_t>(a.logits) % 32 == 0 ? kPairs : kHalves;
  auto kernel = pick_kernel<T, K>(p.threads, loads);
  return launch_clusters(p.n_seg <= kMaxCluster ? p.n_seg : 1, kernel, (unsigned)((a.n_rows + a.concurrent) * p.n_seg), p.threads, 0, a.stream, static_cast<const T*>(a.logits), a.vocab,
                a.row_stride, a.k, p.n_seg, p.chunks_per_seg, a.conf, a.topk_idx, a.topk_prob, a.lse, partials, tickets,
                p.prefetch, a.launch_next, a.concurrent ? (int)a.n_rows : 0);
}

template <typename T>
static cudaError_t dispatch_k(const TopkArgs& a, const TopkPlan& p, void* ws) {
  switch (p.K) {
    case 1: return run_plan<T, 1>(a, p, ws);
    case 2: return run_plan<T, 2>(a, p, ws);
    case 3: return run_plan<T, 3>(a, p, ws);
    case 4: return run_plan<T, 4>(a, p, ws);
    case 6: return run_plan<T, 6>(a, p, ws);
    default: return run_plan<T, 8>(a, p, ws);
  }
}

static int check_shape(int64_t n_rows, int32_t vocab, int32_t k) {
  if (n_rows < 0 || vocab < 1 || k < 1 || k > 8 || k > vocab) return TSD_ERR_INVALID_ARG;
  if (n_rows * (int64_t)kMaxSegments > 0x7fffffffLL) return TSD_ERR_INVALID_ARG;
  // rows longer than kMaxSegments segments of kTopkMaxIter batches (4 Mi fp32 / 8 Mi bf16 logits)
  if ((int64_t)vocab / 4 > (int64_t)kTopkSegChunks * kMaxSegments) return TSD_ERR_INVALID_ARG;
  return TSD_OK;
}

// Everything but the workspace.
static int check_pointers(const TopkArgs& a) {
  int rc = check_shape(a.n_rows, a.vocab, a.k);
  if (rc != TSD_OK) return rc;
  if (a.dtype != TSD_F32 && a.dtype != TSD_BF16) return TSD_ERR_UNSUPPORTED;
  if (a.n_rows == 0) return TSD_OK;
  const int esize = a.dtype == TSD_F32 ? 4 : 2;
  if (!a.logits || !a.conf || !a.topk_idx || !a.topk_prob) return TSD_ERR_INVALID_ARG;
  if (a.row_stride < a.vocab || !aligned16(a.logits) || (a.row_stride * esize) % 16 != 0) return TSD_ERR_INVALID_ARG;
  return TSD_OK;
}

int check_topk(const TopkArgs& a) {
  int rc = check_pointers(a);
  if (rc != TSD_OK || a.n_rows == 0) return rc;
  const size_t need = tsd_confidence_topk_workspace_bytes(a.n_rows, a.vocab, a.k);
  if (need > 0) {  // the documented size is required whichever dtype is passed
    if (!a.workspace || !aligned16(a.workspace)) return TSD_ERR_INVALID_ARG;
    if (a.workspace_bytes < need) return TSD_ERR_WORKSPACE;
  }
  return TSD_OK;
}

int64_t topk_threads(const TopkArgs& a) {
  const TopkPlan p = topk_plan(a.n_rows, a.vocab, a.k, a.dtype == TSD_F32 ? 4 : 8);
  return a.n_rows * p.n_seg * p.threads;
}

int launch_topk(const TopkArgs& a) {
  if (a.n_rows == 0) return TSD_OK;
  const TopkPlan p = topk_plan(a.n_rows, a.vocab, a.k, a.dtype == TSD_F32 ? 4 : 8);
  cudaError_t e = a.dtype == TSD_F32 ? dispatch_k<float>(a, p, a.workspace) : dispatch_k<__nv_bfloat16>(a, p, a.workspace);
  return e != cudaSuccess ? cuda_fail(e, "confidence_topk_kernel") : TSD_OK;
}

}  // namespace tsd

extern "C" {

size_t tsd_confidence_topk_workspace_bytes(int64_t n_rows, int32_t vocab, int32_t k) {
  if (tsd::check_shape(n_rows, vocab, k) != TSD_OK || n_rows == 0) return 0;
  // sized for the narrower element type (more chunks per row can only mean more segments)
  return std::max(tsd::workspace_bytes(n_rows, vocab, k, 8), tsd::workspace_bytes(n_rows, vocab, k, 4));
}

int tsd_confidence_topk(const void* logits, int32_t dtype, int64_t n_rows, int32_t vocab,
                        int64_t row_stride, int32_t k, float* conf, int32_t* topk_idx,
                        float* topk_prob, float* lse, void* workspace, size_t workspace_bytes,
                        uint32_t* status, tsd_stream_t stream) {
  (void)status;
  const tsd::TopkArgs a = {logits, dtype, n_rows, vocab, row_stride, k, conf, topk_idx, topk_prob, lse, workspace,
                           workspace_bytes, stream, tsd::kNextAfter, false};
  int rc = tsd::check_topk(a);
  return rc != TSD_OK ? rc : tsd::launch_topk(a);
}

}  // extern "C"

// ---------------------------------------------------------------------------------------------
// Allocation-free variant.  Some hosts can hand this library nothing but their inputs and outputs:
// an inference-server plug-in whose device memory pool is sized once at start-up and then frozen,
// or a decode loop in which calling cudaMalloc is ruled out because it would stall the whole
// device in the middle of a step.  For them the per-segment partial results and the per-row
// tickets live in a fixed array that is part of the library image: every GPU that loads the
// library carries these bytes until the process exits, which is why the size is kept modest.
namespace tsd {

constexpr size_t kStaticScratchBytes = 1u << 20;  // 1 MiB per device
static __device__ __align__(256) unsigned char g_topk_scratch[kStaticScratchBytes];

// In host code `g_topk_scratch` is only a handle for the runtime, not an address a kernel can use:
// the device address has to be asked for, with the device current.  The lookup is a host-side
// query that allocates nothing; it is repeated on every call rather than remembered, so that the
// address is never one from before a device reset (the first lookup on a device loads the
// library's module there, which is why that first call belongs before any stream capture).
static cudaError_t static_scratch_address(void** out) {
  void* ptr = nullptr;
  cudaError_t e = cudaGetSymbolAddress(&ptr, g_topk_scratch);
  if (e != cudaSuccess) return e;
  *out = ptr;
  return cudaSuccess;
}

}  // namespace tsd

extern "C" size_t tsd_confidence_topk_static_capacity(void) { return tsd::kStaticScratchBytes; }

extern "C" int tsd_confidence_topk_static(const void* logits, int32_t dtype, int64_t n_rows, int32_t vocab,
                                          int64_t row_stride, int32_t k, float* conf, int32_t* topk_idx,
                                          float* topk_prob, float* lse, uint32_t* status,
                                          tsd_stream_t stream) {
  (void)status;
  tsd::TopkArgs a = {logits, dtype, n_rows, vocab, row_stride, k, conf, topk_idx, topk_prob, lse, nullptr, 0, stream, tsd::kNextAfter, false};
  int rc = tsd::check_pointers(a);
  if (rc != TSD_OK || n_rows == 0) return rc;
  // this shape would need more scratch than the library carries: the caller has to use
  // tsd_confidence_topk with a workspace of its own.  The test is on the documented size
  // (tsd_confidence_topk_workspace_bytes, the larger of the two dtypes' needs), so that the check a
  // caller makes beforehand and this one agree.
  if (tsd_confidence_topk_workspace_bytes(n_rows, vocab, k) > tsd::kStaticScratchBytes) return TSD_ERR_WORKSPACE;
  if (tsd::topk_plan(n_rows, vocab, k, dtype == TSD_F32 ? 4 : 8).total_bytes > 0) {
    cudaError_t e = tsd::static_scratch_address(&a.workspace);
    if (e != cudaSuccess) return tsd::cuda_fail(e, "cudaGetSymbolAddress(g_topk_scratch)");
  }
  // ticket words need no clearing (a word that does not carry the in-use tag counts as idle, and
  // the last arrival of a row returns it to idle); the partial-result slots are fully rewritten by
  // every call that reads them
  return tsd::launch_topk(a);
}
