// Stage 1b on CUDA cores: masked verify attention (paper Section 3.3) for the combinations the
// tensor-core kernel does not serve (fp32 inputs) and as a cross-check for it.
//
// One thread block per (sequence, query head, RB draft rows of one branch).  The visible keys (the
// cached tokens, then the rows of every visible draft branch) are cut into chunks of 32 that the
// block's warps take in turn; every warp keeps its own online softmax (maximum, sum, weighted value
// rows) in fp32 registers and the warps meet once, in shared memory, at the end.
//   scores  : D / 8 lanes share a key, each lane holding 8 dimensions of it and of all RB query rows in
//             registers, so a key row is one coalesced read and feeds 8 RB fused multiply-adds per
//             lane; the partial dot products meet in a reduce-scatter (D / 8 - 1 shuffles per
//             group) that leaves every lane with the score of one (key, row) pair.
//   weights : one exponential per (key, row), written to shared memory for the warp.
//   values  : lanes own D / 32 dimensions of the RB output rows; a value row is one coalesced read.
// The kernel before this one gave each lane a whole key (a strided row read per lane, D accumulators per
// lane, one block per branch and head): 184 us for the 288-key case below, 1139 us for 2 x 8 heads x 256
// rows, 800 keys, D = 128, which take 7.4 and 95 us here.
// What bounds it: on the sizes fp32 is used for (checking; a few heads, hundreds of keys) the chain of
// dependent loads and the number of blocks, at larger ones the fp32 pipe (3 of 4 instructions are
// multiply-adds) and the L2 reads of K and V, once per RB rows.  Eight rows of 128 dimensions do not fit the 128 registers that two
// blocks per SM leave a thread: that form spills (fp32 332 bytes of stores and 476 of loads, bf16 368 and 480; the others
// 0 to 28).
#include <limits.h>
#include <math_constants.h>
#include <algorithm>
#include "tsd_common.cuh"

namespace tsd {

constexpr int kRowsChunk = 32;      // keys per chunk
constexpr int kRowsMaxGroups = 1024;  // 32-row groups of a sequence's draft rows at most (256 branches x 128 rows)

// 8 dimensions of a row for lane j of LPK: two 16-byte reads LPK * 16 bytes apart (fp32), or one (bf16).
template <int LPK>
__device__ __forceinline__ void load8(const float* row, int j, float (&x)[8]) {
  const float4 a = *reinterpret_cast<const float4*>(row + 4 * j);
  const float4 b = *reinterpret_cast<const float4*>(row + 4 * (j + LPK));
  x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w;
  x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
}
template <int LPK>
__device__ __forceinline__ void load8(const __nv_bfloat16* row, int j, float (&x)[8]) {
  const uint4 w = *reinterpret_cast<const uint4*>(row + 8 * j);
  const uint32_t u[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    x[2 * i] = __uint_as_float(u[i] << 16);
    x[2 * i + 1] = __uint_as_float(u[i] & 0xffff0000u);
  }
}
// C = 2 or 4 consecutive dimensions of a value row
__device__ __forceinline__ void load_v(const float* p, float (&v)[2]) {
  const float2 a = *reinterpret_cast<const float2*>(p);
  v[0] = a.x; v[1] = a.y;
}
__device__ __forceinline__ void load_v(const float* p, float (&v)[4]) {
  const float4 a = *reinterpret_cast<const float4*>(p);
  v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
}
template <int C>
__device__ __forceinline__ void load_v(const __nv_bfloat16* p, float (&v)[C]) {
#pragma unroll
  for (int i = 0; i < C / 2; ++i) {
    const uint32_t w = reinterpret_cast<const uint32_t*>(p)[i];
    v[2 * i] = __uint_as_float(w << 16);
    v[2 * i + 1] = __uint_as_float(w & 0xffff0000u);
  }
}

template <typename T, int D, int RB, int MAXW>
__global__ void __launch_bounds__(MAXW * 32, RB == 8 ? 2 : 1)
attention_rows_kernel(int S, int B, int R, int Nc, int Hq, int Hkv, int recs_off, int n_qt, int rec_words,
                      const int32_t* __restrict__ mask, const T* __restrict__ q, const T* __restrict__ kc,
                      const T* __restrict__ vc, const T* __restrict__ kd, const T* __restrict__ vd,
                      T* __restrict__ out, float* __restrict__ lse, int64_t qs_b, int64_t qs_r, int64_t qs_h,
                      int64_t cs_b, int64_t cs_r, int64_t cs_h, int64_t ds_b, int64_t ds_r, int64_t ds_h,
                      int64_t os_b, int64_t os_r, int64_t os_h, float sm_scale, uint32_t* __restrict__ status,
                      int concurrent, int next_at_once) {
  constexpr int LPK = D / 8;            // lanes per key
  constexpr int KPI = 32 / LPK;         // keys read at once
  constexpr int SUB = LPK / RB;         // reads per group: SUB * RB scores per key lane, one per lane after the scatter
  constexpr int KG = SUB * KPI;         // keys per group
  constexpr int NG = kRowsChunk / KG;
  constexpr int VC = D / 32;            // value dimensions per lane
  static_assert(LPK % RB == 0, "RB divides D / 8");
  __shared__ int s_vis[kRowsMaxGroups];                                // visible groups of 32 draft rows of this branch
  __shared__ int s_nvis;
  __shared__ __align__(16) float s_p[MAXW][kRowsChunk][RB];            // weights of a warp's chunk
  __shared__ __align__(16) float s_alpha[MAXW][RB];
  __shared__ float s_m[MAXW][RB], s_l[MAXW][RB];
  __shared__ __align__(16) float s_acc[MAXW][RB][D];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
  const int row0 = blockIdx.x * RB, h = blockIdx.y, s = blockIdx.z;
  const int b = row0 / R, g = h / (Hq / Hkv), N = B * R;
  const int j = lane % LPK, slots = kTile / R;
  const unsigned full = 0xffffffffu;
  if (concurrent) {  // beside the kernel before it
    beside_fence();
    settle(mask, q, kc, vc, kd, vd);
  } else {
    grid_wait(mask, q, kc, vc, kd, vd);
  }
  if (next_at_once) grid_launch_beside();

  // the block's query rows, 8 dimensions per lane (requested first: nothing else is needed for them)
  float qr[RB][8];
#pragma unroll
  for (int r = 0; r < RB; ++r) {
    load8<LPK>(q + s * qs_b + (int64_t)(row0 + r) * qs_r + h * qs_h, j, qr[r]);
#pragma unroll
    for (int c = 0; c < 8; ++c) qr[r][c] *= sm_scale;
  }
  // header and cache length, then the query tile's list by the lanes of warp 0
  const bool hdr_ok = mask[H_MAGIC] == kMaskMagic && mask[H_S] == S && mask[H_B] == B && mask[H_R] == R &&
                      mask[H_NC] == Nc;
  const int clen = min(max(mask[kHdrWords + s], 0), Nc);
  if (!hdr_ok) {  // a blob built for another layout: report, write nothing
    if (threadIdx.x == 0 && status) atomicOr(status, TSD_STATUS_BAD_MASK);
    if (concurrent) grid_wait();
    return;
  }
  if (warp == 0) {
    const int32_t* rec = mask + recs_off + (size_t)(s * n_qt + b / slots) * rec_words;
    const int qs = b % slots, n_list = rec_words / 2 - 1, n_entries = min(rec[0], n_list);
    int n = 0;
    for (int e0 = 0; e0 < n_list; e0 += 32) {
      const int e = e0 + lane;
      int kt = 0, nib = 0;
      if (e < n_entries) {
        kt = rec[2 + 2 * e];
        nib = (rec[3 + 2 * e] >> (qs * 2)) & 3;
      }
      int at = __popc(nib);  // inclusive prefix sum of the lanes' counts
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const int o = __shfl_up_sync(full, at, off);
        if (lane >= off) at += o;
      }
      const int total = __shfl_sync(full, at, 31);
      at += n - __popc(nib);
      for (int w = 0; w < 2; ++w)
        if ((nib >> w) & 1) { if (at < kRowsMaxGroups) s_vis[at] = min(kt * 2 + w, N / kRowsChunk - 1); ++at; }
      n += total;
    }
    if (lane == 0) s_nvis = min(n, kRowsMaxGroups);
  }
  __syncthreads();
  const int n_cc = (clen + kRowsChunk - 1) / kRowsChunk, n_chunks = n_cc + s_nvis;

  float m = -CUDART_INF_F, l = 0.f;  // of row lane % RB
  float acc[RB][VC];
#pragma unroll
  for (int r = 0; r < RB; ++r)
#pragma unroll
    for (int c = 0; c < VC; ++c) acc[r][c] = 0.f;

  for (int ch = warp; ch < n_chunks; ch += n_warps) {
    const T *kp, *vp;
    int64_t stride;
    int valid = kRowsChunk;
    if (ch < n_cc) {
      kp = kc + s * cs_b + (int64_t)ch * kRowsChunk * cs_r + g * cs_h;
      vp = vc + s * cs_b + (int64_t)ch * kRowsChunk * cs_r + g * cs_h;
      stride = cs_r;
      valid = min(kRowsChunk, clen - ch * kRowsChunk);
    } else {
      const int64_t row = (int64_t)s_vis[ch - n_cc] * kRowsChunk;
      kp = kd + s * ds_b + row * ds_r + g * ds_h;
      vp = vd + s * ds_b + row * ds_r + g * ds_h;
      stride = ds_r;
    }
    float sc[NG];  // this lane's scores: row lane % RB, keys gi * KG + (j / RB) * KPI + lane / LPK
#pragma unroll
    for (int gi = 0; gi < NG; ++gi) {
      float x[LPK];
#pragma unroll
      for (int u = 0; u < SUB; ++u) {
        const int key = gi * KG + u * KPI + lane / LPK;
        float k8[8];
        load8<LPK>(kp + (int64_t)min(key, valid - 1) * stride, j, k8);
#pragma unroll
        for (int r = 0; r < RB; ++r) {
          float a = 0.f;
#pragma unroll
          for (int c = 0; c < 8; ++c) a = fmaf(qr[r][c], k8[c], a);
          x[u * RB + r] = a;
        }
      }
      // reduce-scatter over the LPK lanes of a key: lane j ends with the sum of x[j]
#pragma unroll
      for (int off = LPK / 2; off >= 1; off >>= 1) {
        const bool upper = j & off;
#pragma unroll
        for (int i = 0; i < off; ++i) {
          const float send = upper ? x[i] : x[i + off], keep = upper ? x[i + off] : x[i];
          x[i] = keep + __shfl_xor_sync(full, send, off);
        }
      }
      sc[gi] = gi * KG + (j / RB) * KPI + lane / LPK < valid ? x[0] : -CUDART_INF_F;
    }
    float mx = sc[0];
#pragma unroll
    for (int gi = 1; gi < NG; ++gi) mx = fmaxf(mx, sc[gi]);
#pragma unroll
    for (int off = RB; off < 32; off <<= 1) mx = fmaxf(mx, __shfl_xor_sync(full, mx, off));
    const float m_new = fmaxf(m, mx);
    const float alpha = m == m_new ? 1.f : expf(m - m_new);  // 0 on the first chunk
    float sum = 0.f;
#pragma unroll
    for (int gi = 0; gi < NG; ++gi) {
      const float p = expf(sc[gi] - m_new);
      s_p[warp][gi * KG + (j / RB) * KPI + lane / LPK][lane % RB] = p;
      sum += p;
    }
#pragma unroll
    for (int off = RB; off < 32; off <<= 1) sum += __shfl_xor_sync(full, sum, off);
    l = l * alpha + sum;
    m = m_new;
    if (lane < RB) s_alpha[warp][lane] = alpha;
    __syncwarp();
#pragma unroll
    for (int r = 0; r < RB; ++r) {
      const float a = s_alpha[warp][r];
#pragma unroll
      for (int c = 0; c < VC; ++c) acc[r][c] *= a;
    }
#pragma unroll 8
    for (int key = 0; key < kRowsChunk; ++key) {
      float v[VC];
      load_v(vp + (int64_t)min(key, valid - 1) * stride + lane * VC, v);  // past the end: weight 0, a readable row
#pragma unroll
      for (int r4 = 0; r4 < RB / 4; ++r4) {
        const float4 p = *reinterpret_cast<const float4*>(&s_p[warp][key][4 * r4]);
#pragma unroll
        for (int c = 0; c < VC; ++c) {
          acc[4 * r4 + 0][c] = fmaf(p.x, v[c], acc[4 * r4 + 0][c]);
          acc[4 * r4 + 1][c] = fmaf(p.y, v[c], acc[4 * r4 + 1][c]);
          acc[4 * r4 + 2][c] = fmaf(p.z, v[c], acc[4 * r4 + 2][c]);
          acc[4 * r4 + 3][c] = fmaf(p.w, v[c], acc[4 * r4 + 3][c]);
        }
      }
    }
    __syncwarp();
  }

  // the warps' parts on a common maximum
  if (lane < RB) { s_m[warp][lane] = m; s_l[warp][lane] = l; }
#pragma unroll
  for (int r = 0; r < RB; ++r)
#pragma unroll
    for (int c = 0; c < VC; ++c) s_acc[warp][r][lane * VC + c] = acc[r][c];
  __syncthreads();
  for (int e = threadIdx.x; e < RB * D; e += blockDim.x) {
    const int r = e / D, c = e % D;
    float M = s_m[0][r];
    for (int w = 1; w < n_warps; ++w) M = fmaxf(M, s_m[w][r]);
    float o = 0.f, lt = 0.f;
    for (int w = 0; w < n_warps; ++w) {
      const float mw = s_m[w][r];
      if (mw == -CUDART_INF_F) continue;  // a warp without keys
      const float f = expf(mw - M);
      lt = fmaf(s_l[w][r], f, lt);
      o = fmaf(s_acc[w][r][c], f, o);
    }
    from_float(out[s * os_b + (int64_t)(row0 + r) * os_r + h * os_h + c], o / lt);
    if (lse && c == 0) lse[((size_t)s * Hq + h) * N + row0 + r] = M + logf(lt);
  }
  if (concurrent) grid_wait();
}

template <typename T, int D, int RB, int MAXW>
static cudaError_t launch_rows(const AttnArgs& a, int warps) {
  const tsd_layout& L = a.L;
  const MaskDims md = mask_dims(L);
  const dim3 grid(L.n_branches * L.rows_per_branch / RB, L.n_q_heads, L.batch);
  return launch(
      attention_rows_kernel<T, D, RB, MAXW>, grid, std::min(warps, MAXW) * 32, 0, a.stream, L.batch, L.n_branches, L.rows_per_branch, L.n_cache, L.n_q_heads, L.n_kv_heads, md.recs_off, md.n_qt,
      md.rec_words, a.mask, static_cast<const T*>(a.q), static_cast<const T*>(a.kc), static_cast<const T*>(a.vc),
      static_cast<const T*>(a.kd), static_cast<const T*>(a.vd), static_cast<T*>(a.out), a.lse, a.qs_b, a.qs_r,
      a.qs_h, a.cs_b, a.cs_r, a.cs_h, a.ds_b, a.ds_r, a.ds_h, a.os_b, a.os_r, a.os_h, a.sm_scale, a.status,
      (int)a.concurrent, (int)a.next_at_once);
}

template <typename T, int D>
static cudaError_t launch_simt(const AttnArgs& a) {
  const tsd_layout& L = a.L;
  const int64_t rows = (int64_t)L.batch * L.n_q_heads * L.n_branches * L.rows_per_branch;
  // As long as 4 rows per block leave no SM with two blocks: 4 rows, and up to 12 warps with a chunk of keys each
  // (4 heads x 128 rows, 288 keys, D = 64: 7.4 us).  Beyond that 8 rows, which halve the reads of K and V, and two
  // blocks of 8 warps per SM (4 heads x 256 rows, 332 keys: 12.8 us; as 4-row blocks in two rounds 14.2 us).
  const int chunks = (L.n_cache + kRowsChunk - 1) / kRowsChunk + L.rows_per_branch / kRowsChunk;
  if (rows <= 4 * 148) return launch_rows<T, D, 4, 12>(a, chunks);
  return launch_rows<T, D, 8, 8>(a, 8);
}

int launch_attention_simt(const AttnArgs& a) {
  cudaError_t e;
  const bool f32 = a.L.dtype == TSD_F32;
  if (a.L.head_dim == 64) e = f32 ? launch_simt<float, 64>(a) : launch_simt<__nv_bfloat16, 64>(a);
  else e = f32 ? launch_simt<float, 128>(a) : launch_simt<__nv_bfloat16, 128>(a);
  if (e != cudaSuccess) return cuda_fail(e, "attention_rows_kernel");
  return TSD_OK;
}

}  // namespace tsd
