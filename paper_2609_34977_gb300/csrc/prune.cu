// MSV-Prune (Sec. 4.1, Eq. 1-3; Alg. 1 stage 1) on the GPU, every tile independently.
//
//   rowstats     a_v = head-mean of the attention (Sec. 4.1.1); 1/||F_l,i|| for every tapped layer
//                (and ||F_l,i||^2, or the log-sum-exp and negentropy of softmax(F_l,i), for the
//                MSE and KL ablations of sim)
//   anchors      top-N_anc of a_v by rank counting of (a_v desc, index asc) keys (Eq. 1), over several
//                CTAs for a long tile; stable lists of anchor and non-anchor tokens by one block scan
//   anchor_sim   a_i = max_p cos(F^L_i, F^L_p) over anchors: 128 x 64 (or 48) register-tiled fp32 products,
//                the feature dimension split over a cluster of 4 or 8 CTAs whose partial tiles are summed
//                in rank order through distributed shared memory; max via atomicMax on
//                order-preserving integer keys (exact, order independent)
//   kmeans       Lloyd on raw F^L of the non-anchor tokens, then the per-cluster, per-layer sums of unit
//                feature rows, the sums of a_j, sizes and Eq. 2 quotas. One thread-block cluster of
//                16 CTAs per tile, each with its slice of the rows in shared memory for every
//                iteration, where they fit and all tiles run at once (kmeans_kernel); the whole GPU,
//                launched cooperatively, for a few larger tiles (kmeans_grid_kernel); one sweep over
//                the rows an iteration for many tiles (kmeans_stream_kernel); clusters of 8 CTAs that
//                re-read the rows from L2 for the shapes none of these takes. Sums across CTAs run in
//                a fixed order
//   scores       s_i = [sum_l w_l f_i . (S_l,k - f_i)] / (|C_k| - 1) + a_i + (A_k - a_i) / (|C_k| - 1),
//                the per-token mean of Eq. 3's S_ij over the other members of its cluster (for
//                the MSE and KL ablations the same cluster-sum identity with raw rows, plus the
//                per-cluster sums of ||F_j||^2 or of the log-sum-exps)
//   select       per cluster the N_k lowest (score, index) keys; kept = anchors + selected, compacted
//                in ascending index order
// Where the rows are resident and the similarity is the cosine, the K-means kernel goes on to the
// scores and the selection itself (fused_select): four launches instead of six.
// All reductions run in a fixed order, so repeated runs give identical bits.
#include <cuda_bf16.h>
#include <math.h>
#include <stdint.h>

#include <cooperative_groups.h>

#include <algorithm>
#include <mutex>
#include <type_traits>

#include "internal.h"
#include "ptx.cuh"
#include "trace.h"

namespace cg = cooperative_groups;

namespace spd {

struct PruneDims {
  int n_tiles, n_tok, off, n, d, L, fin, H, form, n_att, keep, K, iters, n_anc, n_cmp, m;
  int sim;        // SPD_SIM_*
  float wf, wa;   // weights (0 or 1) of the final-layer intra-cluster term and the anchor bracket
  float w[SPD_MAX_FEAT_LAYERS];
  const float* feat[SPD_MAX_FEAT_LAYERS];
};

struct PruneWs {
  float* a_v;       // [T][n]
  float* inv;       // [L][T][n]
  float* st1;       // [L][T][n] MSE: ||F_l,i||^2; KL: log-sum-exp of F_l,i (rounded to fp32)
  float* st2;       // [L][T][n] KL: sum_c P_c log P_c of P = softmax(F_l,i)
  float* st3;       // [L][T][n] KL: log-sum-exp minus its fp32 rounding (st1 + st3 = the fp64 value)
  int8_t* role;     // [T][n] 1 anchor
  int32_t* alist;   // [T][n_anc]
  int32_t* ulist;   // [T][m]
  uint32_t* asim;   // [T][n] ordered keys of a_i
  int32_t* assign;  // [T][m]
  int32_t* counts;  // [T][16]
  int32_t* quotas;  // [T][16]
  float* asum;      // [T][16]
  float* csum;      // [T][L][K][d]
  double* ssum;     // [T][L][16] MSE / KL: per-cluster sums of st1 (+ st3), in fp64
  float* score;     // [T][m]
  int* arrive;      // [T][4] arrivals of a tile's CTAs: anchors, selection, K-means (cleared by rowstats)
  float* gpart;     // K-means over the whole GPU: [T][G][L][K][D] column sums a CTA,
  float* gcent;     // [T][K][D] centroids,
  double* gdsum;    // [T][G][L][16] sums of st1 (+ st3),
  int* gmeta;       // [T][G][32] sizes, flags and a_j sums
  int* status;
};

// The outputs of a prune call (kind, cluster and scores optional).
struct PruneOut {
  int32_t* keep_idx;
  uint8_t* kind;
  int8_t* cluster;
  float* scores;
};

namespace {

__device__ __forceinline__ uint32_t ordered_key(float f) {
  const uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float ordered_val(uint32_t u) {
  return __uint_as_float((u & 0x80000000u) ? (u & 0x7fffffffu) : ~u);
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int off = 16; off; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  return v;
}
__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int off = 16; off; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  return v;
}

// Ranks of list positions [i0, i1) among keys[0..N) (ascending, ties to the lower position): block of
// kRankThreads threads, i1 - i0 <= kRankThreads. keys is padded with the type's largest value to a
// multiple of 16 bytes; rank (shared, [i1 - i0]) receives the counts after a barrier by the caller.
// A lane takes one position and counts the smaller keys with 16-byte broadcast loads, two integer
// instructions a key: the ranking is bound by instruction issue, so 32-bit keys without the index
// are compared where they can be (a tie counts where the other position is lower: <= before the warp's
// positions, < after them). The warps left over split the keys into segments.
constexpr int kRankThreads = 1024;
template <typename T>
__device__ __forceinline__ void count_ranks(const T* keys, int N, int i0, int i1, int* rank) {
  constexpr int V = 16 / int(sizeof(T));
  struct alignas(16) Vec {
    T v[V];
  };
  const Vec* kv = reinterpret_cast<const Vec*>(keys);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int wt = (i1 - i0 + 31) >> 5, nseg = (kRankThreads / 32) / wt;
  for (int i = threadIdx.x; i < i1 - i0; i += kRankThreads) rank[i] = 0;
  __syncthreads();
  const int blk = warp % wt, seg = warp / wt;
  if (seg >= nseg) return;
  const int first = i0 + 32 * blk, i = min(first + lane, i1 - 1);
  const T ki = keys[i];
  const int nv = (N + V - 1) / V, v0 = seg * nv / nseg, v1 = (seg + 1) * nv / nseg;
  const int below = max(v0, min(v1, first / V)), above = max(below, min(v1, (first + 31) / V + 1));
  int cnt[2] = {0, 0};
#pragma unroll 4
  for (int e = v0; e < below; ++e) {
    const Vec x = kv[e];
#pragma unroll
    for (int u = 0; u < V; ++u) cnt[u & 1] += x.v[u] <= ki;
  }
  for (int e = below; e < above; ++e) {
    const Vec x = kv[e];
#pragma unroll
    for (int u = 0; u < V; ++u) cnt[u & 1] += x.v[u] < ki || (x.v[u] == ki && V * e + u < i);
  }
#pragma unroll 4
  for (int e = above; e < v1; ++e) {
    const Vec x = kv[e];
#pragma unroll
    for (int u = 0; u < V; ++u) cnt[u & 1] += x.v[u] < ki;
  }
  if (first + lane < i1) atomicAdd(&rank[i - i0], cnt[0] + cnt[1]);
}
// CTAs that rank one tile's list of n positions: one while its threads suffice, else 128 positions a
// CTA, the last of them to finish going on with the whole list. (2739 keys: 48 us for one CTA sorting
// them, 8 us so; 576 keys: 12.5 us with 64-bit keys, 7 us so.)
__host__ __device__ inline int rank_ctas(int n) { return n <= kRankThreads ? 1 : (n + 127) / 128; }

// True in every thread of the last of the tile's nb CTAs to arrive; what the others wrote before is
// then visible through L2 (__ldcg). The counter was cleared by an earlier kernel of the call.
__device__ __forceinline__ bool last_cta(int* counter, int nb) {
  __shared__ int last;
  if (nb == 1) return true;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(counter, 1) == nb - 1;
  __syncthreads();
  __threadfence();
  return last;
}

// Exclusive prefix sum of one int per thread over a block of 1024 threads.
__device__ int block_scan_excl(int v, int* tmp, int* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int x = v;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, off);
    if (lane >= off) x += y;
  }
  if (lane == 31) tmp[warp] = x;
  __syncthreads();
  if (warp == 0) {
    int w = (lane < (int)(blockDim.x >> 5)) ? tmp[lane] : 0;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, w, off);
      if (lane >= off) w += y;
    }
    tmp[lane] = w;  // inclusive totals of warps
  }
  __syncthreads();
  const int before = (warp ? tmp[warp - 1] : 0) + x - v;
  if (total) *total = tmp[(blockDim.x >> 5) - 1];
  __syncthreads();
  return before;
}

__device__ __forceinline__ const float* feat_row(const PruneDims& p, int l, int t, int i) {
  return p.feat[l] + (size_t(t) * p.n_tok + p.off + i) * p.d;
}

// ---- 1. a_v and inverse norms ---------------------------------------------------------------
template <int SIM>
__global__ void __launch_bounds__(256) rowstats_kernel(PruneDims p, const float* attn,
                                                       PruneWs w) {
  pdl_launch_dependents();
  pdl_wait();
  const int t = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i = blockIdx.x * 8 + warp;
  if (blockIdx.x == 0 && threadIdx.x < 4) w.arrive[4 * t + threadIdx.x] = 0;
  if (i >= p.n) return;
  for (int l = 0; l < p.L; ++l) {
    const float4* r = reinterpret_cast<const float4*>(feat_row(p, l, t, i));
    float ss = 0.0f;
    for (int c = lane; c < p.d / 4; c += 32) {
      const float4 v = r[c];
      ss += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
    }
    ss = warp_sum(ss);
    const size_t o = (size_t(l) * p.n_tiles + t) * p.n + i;
    if (lane == 0) w.inv[o] = 1.0f / sqrtf(ss);
    if (SIM == SPD_SIM_MSE && lane == 0) w.st1[o] = ss;
    if (SIM == SPD_SIM_KL) {
      // softmax over the row in fp64 (z = x - max exact, e^z, sums): the KL scores multiply the
      // log-probabilities by log-ratios of tens, so an fp32 log-sum-exp (about 2e-6 off) would
      // move them by about 1e-4
      float mx = -INFINITY;
      for (int c = lane; c < p.d / 4; c += 32) {
        const float4 v = r[c];
        mx = fmaxf(mx, fmaxf(fmaxf(v.x, v.y), fmaxf(v.z, v.w)));
      }
#pragma unroll
      for (int off = 16; off; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
      double se = 0.0, te = 0.0;
      for (int c = lane; c < p.d / 4; c += 32) {
        const float4 v = r[c];
        const double z[4] = {double(v.x) - mx, double(v.y) - mx, double(v.z) - mx, double(v.w) - mx};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const double e = exp(z[u]);
          se += e;
          te += e * z[u];
        }
      }
      se = warp_sum_d(se);
      te = warp_sum_d(te);
      if (lane == 0) {
        const double lse = double(mx) + log(se);  // log sum_c e^x_c
        const float hi = float(lse);
        w.st1[o] = hi;
        w.st3[o] = float(lse - double(hi));
        w.st2[o] = float(te / se - log(se));      // sum_c P_c log P_c
      }
    }
  }
  if (lane == 0) {
    const int col = (p.form == 0) ? 1 + i : i;
    float s = 0.0f;
    for (int h = 0; h < p.H; ++h) s += attn[(size_t(t) * p.H + h) * p.n_att + col];
    w.a_v[size_t(t) * p.n + i] = s / float(p.H);
  }
}

// ---- 2. anchors (Eq. 1) and stable token lists ------------------------------------------------
__global__ void __launch_bounds__(kRankThreads) anchor_kernel(PruneDims p, PruneWs w) {
  pdl_launch_dependents();
  pdl_wait();
  __shared__ __align__(16) uint32_t keys[4096];
  __shared__ int rank[kRankThreads];
  __shared__ int8_t role[4096];
  __shared__ int tmp[32];
  const int t = blockIdx.y, nb = gridDim.x;
  // a_v descending as ascending keys; ties to the lower index
  for (int i = threadIdx.x; i < ((p.n + 3) & ~3); i += blockDim.x)
    keys[i] = i < p.n ? ~ordered_key(w.a_v[size_t(t) * p.n + i]) : ~0u;
  __syncthreads();
  const int i0 = blockIdx.x * p.n / nb, i1 = (blockIdx.x + 1) * p.n / nb;
  count_ranks(keys, p.n, i0, i1, rank);
  __syncthreads();
  int8_t* grole = w.role + size_t(t) * p.n;
  for (int i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
    role[i] = rank[i - i0] < p.n_anc ? 1 : 0;  // anchor iff its key is among the n_anc smallest
    grole[i] = role[i];
  }
  if (!last_cta(&w.arrive[4 * t], nb)) return;
  if (nb > 1)
    for (int i = threadIdx.x; i < p.n; i += blockDim.x) role[i] = __ldcg(grole + i);
  __syncthreads();
  // stable lists: each thread owns 4 consecutive tokens
  const int base = threadIdx.x * 4;
  int na = 0;
  for (int q = 0; q < 4; ++q)
    if (base + q < p.n) na += role[base + q];
  int ai = block_scan_excl(na, tmp, nullptr), ui = min(base, p.n) - ai;
  // a_i = 0 where the anchor bracket is absent (no anchors, or the ablation without it)
  const uint32_t init = (p.n_anc == 0 || p.wa == 0.0f) ? ordered_key(0.0f) : 0u;
  for (int q = 0; q < 4; ++q) {
    const int i = base + q;
    if (i >= p.n) break;
    if (role[i]) w.alist[size_t(t) * p.n_anc + ai++] = i;
    else w.ulist[size_t(t) * p.m + ui++] = i;
    w.asim[size_t(t) * p.n + i] = init;
  }
}

// Packed pairs of fp32: two IEEE operations an instruction.
__device__ __forceinline__ uint64_t sub_f32x2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t fma_f32x2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t add_f32x2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ float sum_f32x2(uint64_t a) {
  return __uint_as_float(uint32_t(a)) + __uint_as_float(uint32_t(a >> 32));
}

// ---- 3. a_i = max over anchors of cos(F^L_i, F^L_p) -------------------------------------------
// A cluster of AS CTAs per R non-anchor tokens x AW anchors tile, each CTA one slice of the feature
// dimension: 32-wide chunks through shared memory (stored transposed; the next chunk is fetched into
// registers while the current one is multiplied), R / 16 x AW / 16 products a thread. The loop was bound by
// shared-memory reads with 4 x 4 products (16 FMAs per two 16-byte loads: 78 % of the load pipe, 46 % of the
// FMA pipe busy); eight rows a thread (R = 128) halve the loads a product, and the products of two rows go out
// as one packed instruction. Every product is still one fp32 FMA in the order of the features.
// The partial tiles are summed in rank order through distributed shared memory, each CTA finishing R / AS
// rows. AS = 4 at serving batch, 8 where that still leaves at most three CTAs an SM (shorter chains per CTA),
// and R = 64 where R = 128 would leave SMs idle at that. AW is 64, or 48 where that pads the anchors less.
// (64 tiles of 531 x 45 anchors x 1024: 148 -> 115 us; 2260 x 479 x 1280: 98 -> 81 us.)
template <int SIM, int AS, int AW, int kSimRows>
__global__ void __cluster_dims__(AS, 1, 1) __launch_bounds__(256)
    anchor_sim_kernel(PruneDims p, PruneWs w) {
  pdl_launch_dependents();
  pdl_wait();
  constexpr int TJ = AW / 16, TI = kSimRows / 32;  // anchors and row pairs a thread
  constexpr int UP = kSimRows + 4, AP = AW + 4;
  // one buffer: the operand chunks during the products, this CTA's partial dot products after them
  __shared__ __align__(16) float buf[kSimRows * (AW + 1) > 32 * (UP + AP) ? kSimRows * (AW + 1) : 32 * (UP + AP)];
  float(*Us)[UP] = reinterpret_cast<float(*)[UP]>(buf);
  float(*As)[AP] = reinterpret_cast<float(*)[AP]>(buf + 32 * UP);
  float(*P)[AW + 1] = reinterpret_cast<float(*)[AW + 1]>(buf);
  cg::cluster_group cl = cg::this_cluster();
  const int rank = int(cl.block_rank());
  const int t = blockIdx.z, tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int u0 = (blockIdx.x / AS) * kSimRows, p0 = blockIdx.y * AW;
  const int* ul = w.ulist + size_t(t) * p.m;
  const int* al = w.alist + size_t(t) * p.n_anc;
  // staging: warp w loads column dd of rows R / 8 w + i and of anchors AW / 8 w + i
  constexpr int UR = kSimRows / 8, AR = AW / 8;
  const int dd = threadIdx.x & 31, r0 = threadIdx.x >> 5;
  // per-row statistics of the final layer (MSE: squared norms; KL: log-sum-exps, negentropies)
  const size_t so = (size_t(p.fin) * p.n_tiles + t) * p.n;
  constexpr bool kl = SIM == SPD_SIM_KL;
  // rows as 32-bit offsets into the tile's block of F^L (it holds at most 4097 rows of at most 4096 floats), in
  // shared memory (broadcast reads); -1 for rows past the lists
  const float* tile_f = feat_row(p, p.fin, t, -p.off);
  __shared__ int uo[kSimRows], ao[AW];
  // KL: the non-anchor operand is softmax(F^L_i) = exp(F^L_i - lse_i), in fp64
  __shared__ double ulse[kl ? kSimRows : 1];
  if (threadIdx.x < kSimRows) {
    const int r = threadIdx.x;
    const bool uv = u0 + r < p.m;
    uo[r] = uv ? (p.off + ul[u0 + r]) * p.d : -1;
    if (kl) ulse[r] = uv ? double(w.st1[so + ul[u0 + r]]) + double(w.st3[so + ul[u0 + r]]) : 0.0;
  } else if (threadIdx.x < kSimRows + AW) {
    const int r = threadIdx.x - kSimRows;
    ao[r] = p0 + r < p.n_anc ? (p.off + al[p0 + r]) * p.d : -1;
  }
  __syncthreads();
  const int nch = (p.d + 31) / 32, c0 = rank * nch / AS, c1 = (rank + 1) * nch / AS;
  float ru[UR], ra[AR];
  auto fetch = [&](int ch) {
    const int dcol = ch * 32 + dd;
#pragma unroll
    for (int i = 0; i < UR; ++i) {
      const int o = uo[UR * r0 + i];
      const float x = (o >= 0 && dcol < p.d) ? tile_f[o + dcol] : 0.0f;
      if constexpr (kl) ru[i] = (o >= 0 && dcol < p.d) ? float(exp(double(x) - ulse[UR * r0 + i])) : 0.0f;
      else ru[i] = x;
    }
#pragma unroll
    for (int i = 0; i < AR; ++i) {
      const int o = ao[AR * r0 + i];
      ra[i] = (o >= 0 && dcol < p.d) ? tile_f[o + dcol] : 0.0f;
    }
  };
  uint64_t acc[TI][TJ];  // rows 2 (TI ty + i) + {0, 1}, anchors tx + 16 j
#pragma unroll
  for (int i = 0; i < TI; ++i)
#pragma unroll
    for (int j = 0; j < TJ; ++j) acc[i][j] = 0;
  if (c0 < c1) fetch(c0);
  for (int ch = c0; ch < c1; ++ch) {
#pragma unroll
    for (int i = 0; i < UR; i += 4)
      *reinterpret_cast<float4*>(&Us[dd][UR * r0 + i]) = make_float4(ru[i], ru[i + 1], ru[i + 2], ru[i + 3]);
#pragma unroll
    for (int i = 0; i < AR; i += 2) *reinterpret_cast<float2*>(&As[dd][AR * r0 + i]) = make_float2(ra[i], ra[i + 1]);
    __syncthreads();
    if (ch + 1 < c1) fetch(ch + 1);  // in flight during the products below
#pragma unroll 8
    for (int e = 0; e < 32; ++e) {
      uint64_t a[TI];
#pragma unroll
      for (int i = 0; i < TI; i += 2) {
        const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(&Us[e][2 * (TI * ty + i)]);
        a[i] = v.x;
        a[i + 1] = v.y;
      }
#pragma unroll
      for (int j = 0; j < TJ; ++j) {
        const uint32_t bv = __float_as_uint(As[e][tx + 16 * j]);
        const uint64_t b = uint64_t(bv) << 32 | bv;
#pragma unroll
        for (int i = 0; i < TI; ++i) acc[i][j] = fma_f32x2(a[i], b, acc[i][j]);
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < TI; ++i)
#pragma unroll
    for (int j = 0; j < TJ; ++j) {
      P[2 * (TI * ty + i)][tx + 16 * j] = __uint_as_float(uint32_t(acc[i][j]));
      P[2 * (TI * ty + i) + 1][tx + 16 * j] = __uint_as_float(uint32_t(acc[i][j] >> 32));
    }
  cl.sync();
  // rows RPC rank .. RPC rank + RPC - 1 of the tile (TPR threads a row, CPT columns a thread): all
  // AS partials loaded first, summed in rank order
  // (at R = 64, AS = 8 the upper half of the block repeats the lower half's: the maximum stays)
  constexpr int RPC = kSimRows / AS, TPR = RPC < 16 ? 16 : 256 / RPC, CPT = AW / TPR;
  static_assert(AW % TPR == 0, "whole columns a thread");
  const int lr = RPC * rank + int(threadIdx.x) / TPR % RPC, cx = int(threadIdx.x) % TPR;
  float x[AS][CPT];
#pragma unroll
  for (int src = 0; src < AS; ++src) {
    const float* pp = cl.map_shared_rank(&P[0][0], src) + lr * (AW + 1);
#pragma unroll
    for (int j = 0; j < CPT; ++j) x[src][j] = pp[cx + TPR * j];
  }
  const float* inv = w.inv + size_t(p.fin) * p.n_tiles * p.n + size_t(t) * p.n;
  const int ur = u0 + lr;
  float best = -INFINITY;
  // candidates whose maximum over p gives a_i through an increasing map g:
  //   cos: F_i.F_p / (|F_i| |F_p|)             (g = identity)
  //   MSE: 2 F_i.F_p - |F_p|^2                  (g(v) = -(|F_i|^2 - v) / d)
  //   KL:  P_i.F_p - lse_p = -KL(P_i||P_p) + N_i (g(v) = v - N_i)
  if (ur < p.m) {
    const float iu = inv[ul[ur]];
#pragma unroll
    for (int j = 0; j < CPT; ++j) {
      float sdot = 0.0f;
#pragma unroll
      for (int src = 0; src < AS; ++src) sdot += x[src][j];
      const int pa = p0 + cx + TPR * j;
      if (pa < p.n_anc) {
        const int ia = al[pa];
        const float v = SIM == SPD_SIM_COS ? sdot * iu * inv[ia]
                        : SIM == SPD_SIM_MSE ? 2.0f * sdot - w.st1[so + ia]
                                             : float(double(sdot) - double(w.st1[so + ia]) -
                                                     double(w.st3[so + ia]));
        best = fmaxf(best, v);
      }
    }
  }
#pragma unroll
  for (int off = TPR / 2; off; off >>= 1) best = fmaxf(best, __shfl_xor_sync(0xffffffffu, best, off));
  if (cx == 0 && ur < p.m) {
    const int iu = ul[ur];
    if (SIM == SPD_SIM_MSE) best = -(w.st1[so + iu] - best) / float(p.d);
    else if (SIM == SPD_SIM_KL) best = best - w.st2[so + iu];
    atomicMax(&w.asim[size_t(t) * p.n + iu], ordered_key(best));
  }
  cl.sync();  // peers read this CTA's partial tile above
}

// ---- 4. K-means (Lloyd) and Eq. 2 quotas ------------------------------------------------------
// Eq. 2's quotas of K <= 16 clusters (sizes, shared), made to sum to n_cmp, by one whole warp, lane k for
// cluster k; quota [SPD_MAX_CLUSTERS]. All products stay below 2^26. (One thread walking sorted index
// arrays with 64-bit divisions took 3 us on the critical path of every tile, a warp 0.5.)
__device__ __forceinline__ void warp_quotas(const int* sizes, int K, int n_cmp, int* quota) {
  constexpr uint32_t kAll = 0xffffffffu;
  const int k = threadIdx.x & 31;
  const int sz = k < K ? sizes[k] : 0;
  int total = sz;
#pragma unroll
  for (int off = 16; off; off >>= 1) total += __shfl_xor_sync(kAll, total, off);
  const int nonempty = __popc(__ballot_sync(kAll, sz > 0));
  int q = 0;
  if (n_cmp > 0 && total > 0) {
    if (n_cmp < nonempty) {  // one each to the largest clusters, ties to the lower k
      int r = 0;
      for (int j = 0; j < K; ++j) {
        const int sj = __shfl_sync(kAll, sz, j);
        r += sj > sz || (sj == sz && j < k);
      }
      q = sz > 0 && r < n_cmp ? 1 : 0;
    } else {
      const int num = n_cmp * sz, rem = num % total;
      if (sz > 0) q = min(max((2 * num + total) / (2 * total), 1), sz);  // round half away from zero
      int sum = q;
#pragma unroll
      for (int off = 16; off; off >>= 1) sum += __shfl_xor_sync(kAll, sum, off);
      // passes over the clusters, each one up (or down) at most once a pass: in descending fractional part,
      // ties to the lower k (in ascending part, ties to the higher k), among those with room
      while (sum != n_cmp) {
        const bool up = sum < n_cmp;
        const uint32_t room = __ballot_sync(kAll, k < K && (up ? q < sz : q > 1));
        const int need = up ? n_cmp - sum : sum - n_cmp;
        int r = 0;
        for (int j = 0; j < K; ++j) {
          const int rj = __shfl_sync(kAll, rem, j);
          const bool before = up ? (rj > rem || (rj == rem && j < k)) : (rj < rem || (rj == rem && j > k));
          r += (room >> j & 1) && before;
        }
        if ((room >> k & 1) && r < need) q += up ? 1 : -1;
        const int step = min(need, __popc(room));
        sum += up ? step : -step;
        if (step == 0) break;
      }
    }
  }
  if (k < SPD_MAX_CLUSTERS) quota[k] = q;
}

// The fused tail of the K-means kernel: every CTA turns its tokens' accumulated terms into Eq. 3
// scores (as score_kernel) and pushes their (cluster, score, index) keys into every CTA; each CTA
// ranks its own tokens among all non-anchor keys and marks the selected ones in CTA 0, which
// compacts the kept tokens in index order (as select_kernel). keys: 8 (m + 1) + n bytes of every
// CTA's shared memory that nothing else reads any more (the resident rows); j0: this CTA's first
// token of the tile's non-anchor list.
template <int KC>
__device__ void fused_select(const PruneDims& p, const PruneWs& w, const PruneOut& out,
                             cg::cluster_group& cl, int rank, int t, int j0, int nl,
                             const int8_t* asg, const int* idx, const float* av, float* sacc,
                             const int* ncl, const float* ak, uint64_t* keys) {
  const int m = p.m, K = p.K;
  __shared__ int seg[SPD_MAX_CLUSTERS + 1];
  __shared__ int quota[SPD_MAX_CLUSTERS];
  __shared__ int tmp[32];
  uint8_t* kept = reinterpret_cast<uint8_t*>(keys + m + 1);  // CTA 0: [n]
  if (threadIdx.x < 32) {  // every CTA: segment offsets and the Eq. 2 quotas (same in all)
    warp_quotas(ncl, K, p.n_cmp, quota);
    if (threadIdx.x == 0) {
      int acc = 0;
      for (int k = 0; k < K; ++k) {
        seg[k] = acc;
        acc += ncl[k];
      }
      seg[K] = acc;
    }
  }
  __syncthreads();  // every warp's terms of the last layer are in sacc
  uint64_t key[2];  // this thread's tokens jj = threadIdx.x + u blockDim.x (nl <= 2 blockDim.x)
  for (int u = 0; u < 2; ++u) {
    const int jj = threadIdx.x + u * blockDim.x;
    key[u] = ~0ull;
    if (jj < nl) {
      const int k = asg[jj], cnt = ncl[k];
      const float ai = av[jj];
      float s;
      if (cnt <= 1) {
        s = p.wa * 2.0f * ai;
      } else {
        const float inv_c = 1.0f / float(cnt - 1);
        s = sacc[jj] * inv_c + p.wa * (ai + (ak[k] - ai) * inv_c);
      }
      key[u] = (uint64_t(k) << 45) | (uint64_t(ordered_key(s)) << 13) | uint64_t(idx[jj]);
    }
  }
  cl.sync();  // no CTA reads its resident rows any more
  for (int u = 0; u < 2; ++u) {
    const int jj = threadIdx.x + u * blockDim.x;
    if (jj < nl)
      for (int rr = 0; rr < KC; ++rr) cl.map_shared_rank(keys, rr)[j0 + jj] = key[u];
  }
  if (rank == 0)
    for (int i = threadIdx.x; i < p.n; i += blockDim.x) kept[i] = uint8_t(w.role[size_t(t) * p.n + i]);
  cl.sync();  // every CTA holds all m keys; CTA 0 the anchor flags
  uint8_t* kept0 = cl.map_shared_rank(kept, 0);
  // rank of each of this CTA's tokens among all keys: eight lanes a token, every eighth key each
  for (int jb = 0; jb < nl; jb += int(blockDim.x) / 8) {
    const int jj = jb + int(threadIdx.x) / 8;
    const uint64_t ki = keys[j0 + min(jj, nl - 1)];
    int r = 0;
#pragma unroll 4
    for (int j = threadIdx.x & 7; j < m; j += 8) r += keys[j] < ki;
#pragma unroll
    for (int off = 4; off; off >>= 1) r += __shfl_xor_sync(0xffffffffu, r, off);
    if ((threadIdx.x & 7) == 0 && jj < nl) {
      const int k = int(ki >> 45);
      // the key at sorted position r of cluster k's segment is kept iff r - seg[k] < quota[k]
      if (r - seg[k] < quota[k]) kept0[ki & 0x1fffu] = 2;
      if (out.cluster) out.cluster[size_t(t) * p.n + (ki & 0x1fffu)] = int8_t(k);
      if (out.scores) out.scores[size_t(t) * p.n + (ki & 0x1fffu)] = ordered_val(uint32_t(ki >> 13));
    }
  }
  cl.sync();  // the selected flags are in CTA 0
  if (rank != 0) return;
  // compaction in index order: thread th owns tokens [th q, th q + q)
  const int q = (p.n + blockDim.x - 1) / blockDim.x, base = threadIdx.x * q;
  int nk = 0;
  for (int u = 0; u < q; ++u)
    if (base + u < p.n) nk += kept[base + u] != 0;
  int pos = block_scan_excl(nk, tmp, nullptr);
  for (int u = 0; u < q; ++u) {
    const int i = base + u;
    if (i >= p.n) break;
    if (kept[i]) {
      if (pos < p.keep) out.keep_idx[size_t(t) * p.keep + pos] = i;
      else set_status(w.status, SPD_EINVAL);
      ++pos;
    }
    if (out.kind) out.kind[size_t(t) * p.n + i] = kept[i];
    if (kept[i] == 1) {
      if (out.cluster) out.cluster[size_t(t) * p.n + i] = -1;
      if (out.scores) out.scores[size_t(t) * p.n + i] = INFINITY;
    }
  }
}

// Row jj of this CTA's tokens: resident in shared memory (rows + jj D) or in global memory
// (g + (row0 + idx[jj]) D), optionally scaled by scale[jj].
struct RowAccess {
  const float* rows;  // resident rows, or null
  const float* g;
  size_t row0;
  const int* idx;
  int D;
  const float* scale;  // or null
  __device__ __forceinline__ const float* row(int jj) const {
    return rows ? rows + size_t(jj) * D : g + (row0 + idx[jj]) * D;
  }
  __device__ __forceinline__ float4 v4(int jj, int c) const {
    float4 v = *reinterpret_cast<const float4*>(row(jj) + c);
    if (scale) {
      const float sc = scale[jj];
      v.x *= sc;
      v.y *= sc;
      v.z *= sc;
      v.w *= sc;
    }
    return v;
  }
};

// This CTA's nl <= 1024 tokens listed by cluster, in token order within each: ord[start[k] .. start[k + 1]).
// A warp a cluster (ballots over 32 tokens at a time); every thread of the block calls it, and a barrier
// before the lists are read is the caller's.
__device__ __forceinline__ void cluster_lists(const int8_t* asg, int nl, int K, int* cnt, uint16_t* ord, int* start) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int k = warp; k < K; k += nw) {
    int n = 0;
    for (int b = 0; b < nl; b += 32) n += __popc(__ballot_sync(0xffffffffu, b + lane < nl && asg[b + lane] == k));
    if (lane == 0) cnt[k] = n;
  }
  __syncthreads();
  for (int k = warp; k < K; k += nw) {
    int at = 0;
    for (int j = 0; j < k; ++j) at += cnt[j];
    if (lane == 0) {
      start[k] = at;
      if (k == K - 1) start[K] = nl;
    }
    for (int b = 0; b < nl; b += 32) {
      const bool mine = b + lane < nl && asg[b + lane] == k;
      const uint32_t who = __ballot_sync(0xffffffffu, mine);
      if (mine) ord[at + __popc(who & ((1u << lane) - 1))] = uint16_t(b + lane);
      at += __popc(who);
    }
  }
}

// part[k][c] = sum over this CTA's tokens of cluster k, in token order, of value.v4(token, c): four
// adjacent columns a thread, eight rows in flight. The rows come sorted by cluster, so a row costs one load
// and four additions (with a running sum for each of the K clusters it was 16 predicated additions).
__device__ __forceinline__ void column_sums(float* part, int K, int D, int nl, const uint16_t* ord, const int* start,
                                            RowAccess value) {
  for (int c = 4 * threadIdx.x; c < D; c += 4 * blockDim.x)
    for (int k = 0; k < K; ++k) {
      const int j1 = start[k + 1];
      float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
      for (int jb = start[k]; jb < j1; jb += 8) {
        float4 xv[8];
#pragma unroll
        for (int u = 0; u < 8; ++u)
          xv[u] = jb + u < j1 ? value.v4(ord[jb + u], c) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          acc.x += xv[u].x;
          acc.y += xv[u].y;
          acc.z += xv[u].z;
          acc.w += xv[u].w;
        }
      }
      *reinterpret_cast<float4*>(part + k * D + c) = acc;
    }
}

// The nearest of four centroids for each of RP rows from the lanes' packed partial distances.
template <int RP>
__device__ __forceinline__ void assign4_nearest(const uint64_t (&acc)[RP][4], int n, bool first, int8_t* asg,
                                                int* changed) {
  constexpr int NV = 4 * RP;
  const int lane = threadIdx.x & 31;
  float v[NV];
#pragma unroll
  for (int i = 0; i < RP; ++i)
#pragma unroll
    for (int k = 0; k < 4; ++k) v[4 * i + k] = sum_f32x2(acc[i][k]);
  int off = 16;
#pragma unroll
  for (int h = NV / 2; h >= 1; h >>= 1, off >>= 1) {
    const bool up = lane & off;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const float recv = __shfl_xor_sync(0xffffffffu, up ? v[i] : v[i + h], off);
      v[i] = (up ? v[i + h] : v[i]) + recv;
    }
  }
  const int low = off;  // lanes that differ below 2 low hold the same value's parts
  for (; off; off >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], off);
  // value index = lane / (2 low) = 4 row + k: the nearest centroid, ties to the lower k (a NaN distance loses,
  // but wins at k = 0, as in a scan over k that replaces the first distance by smaller ones)
  int best = (lane / (2 * low)) & 3;
  if (v[0] != v[0]) v[0] = best == 0 ? -INFINITY : INFINITY;
#pragma unroll
  for (int s = 1; s <= 2; s <<= 1) {
    const float od = __shfl_xor_sync(0xffffffffu, v[0], 2 * low * s);
    const int ob = __shfl_xor_sync(0xffffffffu, best, 2 * low * s);
    if (od < v[0] || (od == v[0] && ob < best)) {
      v[0] = od;
      best = ob;
    }
  }
  const int jj = lane / (8 * low);
  if (lane % (8 * low) == 0 && jj < n) {
    if (first || asg[jj] != best) *changed = 1;
    asg[jj] = int8_t(best);
  }
}

// assign_rows for K = 4, the calling warp's next n (at most RP count) rows at a time: a centroid's 16 bytes
// serve RP rows, differences and squares are packed, and the 4 RP partial distances are summed over the lanes
// by halving exchanges (lane bits 4, 3, ... pick the value) instead of a butterfly each. The loop is bound by
// issue: about 155 instructions a row of 1024 at RP = 4 where a row at a time took about 450 (28 rows of a CTA
// of eight warps: 4.3 -> 2.0 us).
template <int RP, typename Row>
__device__ __forceinline__ void assign4_rows(const float* cent, int D, int n, bool first, int8_t* asg, int* changed,
                                             Row xrow) {
  const int lane = threadIdx.x & 31;
  const float* x[RP];
#pragma unroll
  for (int i = 0; i < RP; ++i) x[i] = xrow(min(i, n - 1));
  uint64_t acc[RP][4];
#pragma unroll
  for (int i = 0; i < RP; ++i)
#pragma unroll
    for (int k = 0; k < 4; ++k) acc[i][k] = 0;
#pragma unroll 2
  for (int c = 4 * lane; c < D; c += 128) {
    ulonglong2 xv[RP], cv[4];
#pragma unroll
    for (int i = 0; i < RP; ++i) xv[i] = *reinterpret_cast<const ulonglong2*>(x[i] + c);
#pragma unroll
    for (int k = 0; k < 4; ++k) cv[k] = *reinterpret_cast<const ulonglong2*>(cent + k * D + c);
#pragma unroll
    for (int i = 0; i < RP; ++i)
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const uint64_t d0 = sub_f32x2(xv[i].x, cv[k].x), d1 = sub_f32x2(xv[i].y, cv[k].y);
        acc[i][k] = fma_f32x2(d0, d0, acc[i][k]);
        acc[i][k] = fma_f32x2(d1, d1, acc[i][k]);
      }
  }
  assign4_nearest<RP>(acc, n, first, asg, changed);
}
// The same with the centroids in the caller's registers: lane's columns 4 lane + 128 j of centroid k in cr[k][j].
template <int RP, typename Row>
__device__ __forceinline__ void assign4_regs(const ulonglong2 (&cr)[4][8], int D, int n, bool first, int8_t* asg,
                                             int* changed, Row xrow) {
  const int lane = threadIdx.x & 31;
  const float* x[RP];
#pragma unroll
  for (int i = 0; i < RP; ++i) x[i] = xrow(min(i, n - 1));
  uint64_t acc[RP][4];
#pragma unroll
  for (int i = 0; i < RP; ++i)
#pragma unroll
    for (int k = 0; k < 4; ++k) acc[i][k] = 0;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int c = 4 * lane + 128 * j;
#pragma unroll
    for (int i = 0; i < RP; ++i) {
      const ulonglong2 xv = c < D ? *reinterpret_cast<const ulonglong2*>(x[i] + c) : make_ulonglong2(0, 0);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const uint64_t d0 = sub_f32x2(xv.x, cr[k][j].x), d1 = sub_f32x2(xv.y, cr[k][j].y);
        acc[i][k] = fma_f32x2(d0, d0, acc[i][k]);
        acc[i][k] = fma_f32x2(d1, d1, acc[i][k]);
      }
    }
  }
  assign4_nearest<RP>(acc, n, first, asg, changed);
}
// ... of all nl rows by the block's warps.
template <int RP, typename Row>
__device__ __forceinline__ void assign4(const float* cent, int D, int nl, bool first, int8_t* asg, int* changed,
                                        Row xrow) {
  const int nw = blockDim.x >> 5;
  for (int jb = (threadIdx.x >> 5) * RP; jb < nl; jb += nw * RP)
    assign4_rows<RP>(cent, D, nl - jb, first, asg + jb, changed, [&](int i) { return xrow(jb + i); });
}

// Nearest centroid (squared Euclidean, ties to the lower cluster) of each of this CTA's nl rows, one
// warp a row; *changed is raised where an assignment differs from asg's (or `first`).
template <int KN, typename Row>
__device__ __forceinline__ void assign_rows(const float* cent, int K, int D, int nl, bool first, int8_t* asg,
                                            int* changed, Row xrow) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  if constexpr (KN == 4) {  // as many rows at a time as leave no warp idle
    if (nl > 2 * nw) assign4<4>(cent, D, nl, first, asg, changed, xrow);
    else if (nl > nw) assign4<2>(cent, D, nl, first, asg, changed, xrow);
    else assign4<1>(cent, D, nl, first, asg, changed, xrow);
  } else {
    for (int jj = warp; jj < nl; jj += nw) {
      const float* x = xrow(jj);
      float part_d[KN];
#pragma unroll
      for (int k = 0; k < KN; ++k) part_d[k] = 0.0f;
      // 16-byte loads, four in flight per lane (D is a multiple of 4)
      for (int cb = 4 * lane; cb < D; cb += 512) {
        float4 xv[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int c = cb + 128 * u;
          xv[u] = c < D ? *reinterpret_cast<const float4*>(x + c) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int c = cb + 128 * u;
          if (c < D) {
#pragma unroll
            for (int k = 0; k < KN; ++k)
              if (k < K) {
                const float4 ce = *reinterpret_cast<const float4*>(cent + k * D + c);
                const float d0 = xv[u].x - ce.x, d1 = xv[u].y - ce.y, d2 = xv[u].z - ce.z,
                            d3 = xv[u].w - ce.w;
                part_d[k] += d0 * d0 + d1 * d1 + d2 * d2 + d3 * d3;
              }
          }
        }
      }
      int best = 0;
      float bd = 0.0f;
#pragma unroll
      for (int k = 0; k < KN; ++k)
        if (k < K) {
          const float dk = warp_sum(part_d[k]);
          if (k == 0 || dk < bd) {
            bd = dk;
            best = k;
          }
        }
      if (lane == 0) {
        if (first || asg[jj] != best) *changed = 1;
        asg[jj] = int8_t(best);
      }
    }
  }
}

// Sums over the KC CTAs of the cluster, in rank order, of the per-CTA column sums `part` (K x D in
// every CTA's shared memory), for this CTA's slice of columns; `emit(k, c, four values)` consumes them.
template <int KC, typename F>
__device__ __forceinline__ void cluster_column_reduce(cg::cluster_group& cl, float* part, int K, int D,
                                                      int rank, F emit) {
  const int n4 = D / 4, c0 = rank * n4 / KC, c1 = (rank + 1) * n4 / KC, width = c1 - c0;  // 16-byte columns
  for (int e = threadIdx.x; e < K * width; e += blockDim.x) {
    const int k = e / width, c = 4 * (c0 + e - k * width);
    float4 x[KC];
#pragma unroll
    for (int rr = 0; rr < KC; ++rr)  // in flight
      x[rr] = *reinterpret_cast<const float4*>(cl.map_shared_rank(part, rr) + k * D + c);
    float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int rr = 0; rr < KC; ++rr) {
      sum.x += x[rr].x;
      sum.y += x[rr].y;
      sum.z += x[rr].z;
      sum.w += x[rr].w;
    }
    emit(k, c, sum);
  }
}

// K-means over one tile per cluster of KC CTAs, CTA r owning the non-anchor tokens
// [r m / KC, (r+1) m / KC). RES: those tokens' F^L rows are copied into the CTA's shared memory
// once (one bulk copy per row) and every Lloyd iteration reads them there; otherwise each
// iteration re-reads them from global memory (L2). KN: an upper bound of K known at compile time
// (K itself for the paper's K = 4), sizing the per-thread accumulators.
template <int KN>
constexpr int kmeans_threads() { return KN == 4 ? 256 : 512; }

// COS: the similarity kind is the cosine (the paper's); the MSE / KL ablations' extra sums are
// compiled into the other instance only (the Lloyd loop is instruction-bound).
// FUSED (RES and COS only): the kernel goes on to the Eq. 3 scores of its tokens, from the resident
// rows of each layer and that layer's cluster sums pushed into every CTA, and the rank-0 CTA then
// selects and compacts the kept tokens (the work of score_kernel and select_kernel, without their
// launches and without reading the features again).
template <int KC, bool RES, int KN, bool COS, bool FUSED = false>
__global__ void __launch_bounds__(kmeans_threads<KN>()) kmeans_kernel(PruneDims p, PruneWs w,
                                                                       PruneOut out) {
  static_assert(!FUSED || (RES && COS), "the fused tail reads resident rows of unit-norm scores");
  pdl_launch_dependents();
  pdl_wait();
  extern __shared__ __align__(16) float ksm[];
  const int K = p.K, D = p.d, m = p.m;
  const int nl_max = (m + KC - 1) / KC;
  float* rows = ksm;                                          // RES: [nl_max][D]
  float* cent = ksm + (RES ? size_t(nl_max) * D : size_t(0));  // [K][D] centroids (every CTA)
  float* part = cent + size_t(K) * D;                         // [K][D] this CTA's column sums
  __shared__ int cnt[SPD_MAX_CLUSTERS];   // this CTA's cluster sizes
  __shared__ float asum_part[SPD_MAX_CLUSTERS];
  __shared__ double ssum_part[SPD_MAX_CLUSTERS];  // MSE / KL: this CTA's sums of st1 (+ st3) per cluster
  __shared__ int changed;      // this CTA's assignment changed in the current iteration
  __shared__ int any_changed;  // ... some CTA's of the cluster
  __shared__ int8_t asg[4096 / KC + 1];
  __shared__ uint16_t ord[4096 / KC + 1];       // this CTA's tokens by cluster
  __shared__ int start[SPD_MAX_CLUSTERS + 1];   // ... the clusters' first positions in ord
  __shared__ int idx[4096 / KC + 1];     // patch index of each of this CTA's tokens
  __shared__ float av[4096 / KC + 1];    // their a_j
  __shared__ float rinv[4096 / KC + 1];  // their 1 / ||F_l,j|| (cos) or st1 (MSE, KL) of the layer
  __shared__ int ncl[SPD_MAX_CLUSTERS];  // cluster sizes over the whole cluster of CTAs
  __shared__ float ak[SPD_MAX_CLUSTERS];  // FUSED: the cluster's sums of a_j (rank order)
  __shared__ float sacc[FUSED ? 4096 / KC + 1 : 1];  // FUSED: per token, sum_l w_l f_i.(S_l,k - f_i)
  __shared__ uint64_t rows_bar;
  cg::cluster_group cl = cg::this_cluster();
  const int rank = int(cl.block_rank());
  const int t = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nw = blockDim.x >> 5;
  const int j0 = rank * m / KC, j1 = (rank + 1) * m / KC, nl = j1 - j0;
  const int* ul = w.ulist + size_t(t) * m;
  const size_t row0 = size_t(t) * p.n_tok + p.off;  // feature row of patch 0 of this tile
  const float* fin = p.feat[p.fin];
  if (threadIdx.x < SPD_MAX_CLUSTERS) ncl[threadIdx.x] = 0;
  for (int jj = threadIdx.x; jj < nl; jj += blockDim.x) {
    idx[jj] = ul[j0 + jj];
    av[jj] = ordered_val(w.asim[size_t(t) * p.n + ul[j0 + jj]]);
  }
  if (RES && threadIdx.x == 0) {
    mbar_init(&rows_bar, 1);
    fence_mbar_init();
  }
  __syncthreads();
  // the rows and, in the same phase of the barrier, the seeds (a CTA without tokens loads the seeds too)
  if (RES && m > 0 && warp == 0) {
    if (lane == 0) mbar_arrive_expect_tx(&rows_bar, uint32_t(nl + K) * D * 4);
    __syncwarp();
    for (int k = lane; k < K; k += 32)
      bulk_load(cent + size_t(k) * D, fin + (row0 + ul[(k * m) / K]) * D, uint32_t(D) * 4, &rows_bar);
    for (int jj = lane; jj < nl; jj += 32)
      bulk_load(rows + size_t(jj) * D, fin + (row0 + idx[jj]) * D, uint32_t(D) * 4, &rows_bar);
  }
  if (!RES && m > 0) {
#pragma unroll 4
    for (int e = threadIdx.x; e < K * D; e += blockDim.x) {
      const int k = e / D, c = e % D;
      cent[e] = feat_row(p, p.fin, t, ul[(k * m) / K])[c];
    }
  }
  if (RES && m > 0) {
    volatile int no_abort = 0;
    if (!mbar_wait(&rows_bar, 0, &no_abort, kWaitBudget)) {
      set_status(w.status, SPD_ETIMEOUT);
      mbar_wait(&rows_bar, 0, &no_abort, kWaitBudget);  // the copies land before anything reuses it
    }
  }
  __syncthreads();
  // this CTA's token jj of the tile's non-anchor list, row of F^L
  auto xrow = [&](int jj) -> const float* {
    return RES ? rows + size_t(jj) * D : fin + (row0 + idx[jj]) * D;
  };
  for (int it = 0; it < p.iters && m > 0; ++it) {
    // assignment of this CTA's points
    if (threadIdx.x == 0) changed = 0;
    __syncthreads();
    assign_rows<KN>(cent, K, D, nl, it == 0, asg, &changed, xrow);
    if (!RES && it > 0) {
      // the column sums are another pass over the rows in L2: not for an assignment that repeats
      cl.sync();
      if (warp == 0) {
        const int any = __any_sync(0xffffffffu, lane < KC && *cl.map_shared_rank(&changed, lane) != 0);
        if (lane == 0) any_changed = any;
      }
      __syncthreads();
      if (!any_changed) {
        cl.sync();  // every CTA has read the flags
        break;      // cluster-uniform decision
      }
    }
    __syncthreads();
    // this CTA's column sums (token order, in registers) and sizes
    cluster_lists(asg, nl, K, cnt, ord, start);
    __syncthreads();
    column_sums(part, K, D, nl, ord, start, RowAccess{RES ? rows : nullptr, fin, row0, idx, D, nullptr});
    cl.sync();
    // one warp reads the peers' flags and sizes (lane r: CTA r) and publishes them in this CTA
    if (warp == 0) {
      const int f = lane < KC ? *cl.map_shared_rank(&changed, lane) : 0;
      const int any = __any_sync(0xffffffffu, f != 0);
      for (int k = 0; k < K; ++k) {
        int n = lane < KC ? cl.map_shared_rank(cnt, lane)[k] : 0;
#pragma unroll
        for (int off = 16; off; off >>= 1) n += __shfl_xor_sync(0xffffffffu, n, off);
        if (lane == 0) ncl[k] = n;
      }
      if (lane == 0) any_changed = any;
    }
    __syncthreads();
    if (it > 0 && !any_changed) break;  // cluster-uniform decision
    // new centroids for this CTA's column slice, written into every CTA
    cluster_column_reduce<KC>(cl, part, K, D, rank, [&](int k, int c, float4 v) {
      const float n = float(ncl[k]);
      if (n > 0.0f) v = make_float4(v.x / n, v.y / n, v.z / n, v.w / n);
      else v = *reinterpret_cast<const float4*>(cent + k * D + c);
      for (int rr = 0; rr < KC; ++rr) *reinterpret_cast<float4*>(cl.map_shared_rank(cent, rr) + k * D + c) = v;
    });
    cl.sync();
  }
  // final assignment (lists and sizes are its: an assignment that repeats leaves them as they were): the
  // per-cluster sums of a_j in token order, and the assignment itself
  __syncthreads();
  if (m == 0) {
    cluster_lists(asg, nl, K, cnt, ord, start);
    __syncthreads();
  }
  if (!FUSED)
    for (int jj = threadIdx.x; jj < nl; jj += blockDim.x) w.assign[size_t(t) * m + j0 + jj] = asg[jj];
  if (threadIdx.x < K) {
    float a = 0.0f;
    for (int j = start[threadIdx.x]; j < start[threadIdx.x + 1]; ++j) a += av[ord[j]];
    asum_part[threadIdx.x] = a;
  }
  // per layer: sums over each cluster of unit feature rows (F_l,j / ||F_l,j||), or of raw rows and
  // of st1 for the MSE and KL similarities
  // (RES: the final layer first, from the resident rows; then each other layer's rows are copied
  // into the same buffer)
  constexpr bool cos_sim = COS;
  for (int li = 0; li < p.L; ++li) {
    const int l = RES ? (li == 0 ? p.fin : (li <= p.fin ? li - 1 : li)) : li;
    const float* rstat = (cos_sim ? w.inv : w.st1) + (size_t(l) * p.n_tiles + t) * p.n;
    const float* fl = p.feat[l];
    __syncthreads();  // the previous layer's rows are no longer read
    for (int jj = threadIdx.x; jj < nl; jj += blockDim.x) rinv[jj] = rstat[idx[jj]];
    if (RES && l != p.fin && warp == 0 && nl > 0) {
      if (lane == 0) mbar_arrive_expect_tx(&rows_bar, uint32_t(nl) * D * 4);
      __syncwarp();
      for (int jj = lane; jj < nl; jj += 32)
        bulk_load(rows + size_t(jj) * D, fl + (row0 + idx[jj]) * D, uint32_t(D) * 4, &rows_bar);
    }
    if (RES && l != p.fin && nl > 0) {
      volatile int no_abort = 0;
      if (!mbar_wait(&rows_bar, li & 1, &no_abort, kWaitBudget)) {
        set_status(w.status, SPD_ETIMEOUT);
        mbar_wait(&rows_bar, li & 1, &no_abort, kWaitBudget);
      }
    }
    __syncthreads();
    if (!cos_sim && threadIdx.x == 0) {  // token order, fp64 (KL: the fp64 log-sum-exps)
      const float* lo = p.sim == SPD_SIM_KL ? w.st3 + (size_t(l) * p.n_tiles + t) * p.n : nullptr;
      for (int k = 0; k < K; ++k) ssum_part[k] = 0.0;
      for (int jj = 0; jj < nl; ++jj)
        ssum_part[asg[jj]] += double(rinv[jj]) + (lo ? double(lo[idx[jj]]) : 0.0);
    }
    column_sums(part, K, D, nl, ord, start,
                RowAccess{RES ? rows : nullptr, fl, row0, idx, D, cos_sim ? rinv : static_cast<float*>(nullptr)});
    cl.sync();
    float* csum = w.csum + (size_t(t) * p.L + l) * K * D;
    cluster_column_reduce<KC>(cl, part, K, D, rank, [&](int k, int c, float4 sum) {
      if constexpr (FUSED) {  // the layer's cluster sums into every CTA (the centroids are done)
        for (int rr = 0; rr < KC; ++rr) *reinterpret_cast<float4*>(cl.map_shared_rank(cent, rr) + k * D + c) = sum;
      } else {
        *reinterpret_cast<float4*>(csum + k * D + c) = sum;
      }
    });
    if (!cos_sim && rank == 0 && warp == 1) {  // CTA sums added in rank order
      for (int k = 0; k < K; ++k) {
        const double sr = lane < KC ? cl.map_shared_rank(ssum_part, lane)[k] : 0.0;
        double a = 0.0;
        for (int rr = 0; rr < KC; ++rr) a += __shfl_sync(0xffffffffu, sr, rr);
        if (lane == 0) w.ssum[(size_t(t) * p.L + l) * 16 + k] = a;
      }
    }
    if (FUSED && li == p.L - 1 && warp == 2) {
      // every CTA: the cluster's sums of a_j over the CTAs, in rank order (lane r reads CTA r)
      float ar[SPD_MAX_CLUSTERS];  // all of CTA lane's sums first (one remote round trip)
      const float* peer = lane < KC ? cl.map_shared_rank(asum_part, lane) : nullptr;
      for (int k = 0; k < K; ++k) ar[k] = peer ? peer[k] : 0.0f;
      for (int k = 0; k < K; ++k) {
        float a = 0.0f;
        for (int rr = 0; rr < KC; ++rr) a += __shfl_sync(0xffffffffu, ar[k], rr);
        if (lane == 0) ak[k] = a;
      }
    }
    if (!FUSED && li == p.L - 1 && rank == 0 && warp == 0) {
      // sizes and a_j sums over the CTAs (lane r reads CTA r; the a_j sums added in rank order)
      for (int k = 0; k < K; ++k) {
        const float ar = lane < KC ? cl.map_shared_rank(asum_part, lane)[k] : 0.0f;
        int n = lane < KC ? cl.map_shared_rank(cnt, lane)[k] : 0;
#pragma unroll
        for (int off = 16; off; off >>= 1) n += __shfl_xor_sync(0xffffffffu, n, off);
        float a = 0.0f;
        for (int rr = 0; rr < KC; ++rr) a += __shfl_sync(0xffffffffu, ar, rr);
        if (lane == 0) {
          ncl[k] = n;
          w.counts[t * 16 + k] = n;
          w.asum[t * 16 + k] = a;
        }
      }
      __syncwarp();
      warp_quotas(ncl, K, p.n_cmp, w.quotas + t * 16);
    }
    cl.sync();  // peers' shared memory is read above; keep it alive and unchanged until here
    if constexpr (FUSED) {
      // this CTA's tokens: f_i.(S_l,k - f_i) with f = F / |F| from the resident rows of layer l
      const float wl = (l == p.fin) ? p.wf : p.w[l];
      for (int jj = warp; jj < nl; jj += nw) {
        if (li == 0 && lane == 0) sacc[jj] = 0.0f;
        if (wl == 0.0f) continue;
        const float* x = rows + size_t(jj) * D;
        const float* sk = cent + size_t(asg[jj]) * D;
        const float iv = rinv[jj];
        float dot = 0.0f;
        for (int c = 4 * lane; c < D; c += 128) {
          const float4 xv = *reinterpret_cast<const float4*>(x + c);
          const float4 sv = *reinterpret_cast<const float4*>(sk + c);
          const float b0 = xv.x * iv, b1 = xv.y * iv, b2 = xv.z * iv, b3 = xv.w * iv;
          dot += b0 * (sv.x - b0) + b1 * (sv.y - b1) + b2 * (sv.z - b2) + b3 * (sv.w - b3);
        }
        dot = warp_sum(dot);
        if (lane == 0) sacc[jj] += wl * dot;
      }
    }
  }
  if constexpr (FUSED) fused_select<KC>(p, w, out, cl, rank, t, j0, nl, asg, idx, av, sacc, ncl, ak,
                                        reinterpret_cast<uint64_t*>(rows));
}

// ---- 4b. K-means of a few large tiles over the whole GPU -----------------------------------------
// G CTAs per tile (all resident: a cooperative launch of at most one CTA an SM), CTA r owning the
// non-anchor tokens [r m / G, (r+1) m / G), whose F^L rows it keeps in shared memory where they fit. A
// cluster holds at most 16 CTAs, so one image of thousands of tokens (11.5 MB of rows at 2260 x 1280)
// ran on 8 SMs that read every row from L2 twice an iteration: 522 us. Here an iteration is the
// assignment, the column sums (per-CTA, in token order) to L2, a barrier over the tile's CTAs, each
// CTA's share of the columns summed over the CTAs in a fixed order, a second barrier and the new
// centroids back: bound by the two barriers and the L2 round trips behind them (about 8 us), no longer by
// the rows.
constexpr int kGridThreads = 512;
constexpr int kGridMaxCtas = 160;  // all tiles (workspace)
constexpr int kGridMaxRows = 512;  // a CTA
// Ints a CTA: [0, 16) its clusters' sizes, the CTA's changed flag in bit 30 of each; [16, 32) the a_j sums as
// float bits.
constexpr int kGridMeta = 2 * SPD_MAX_CLUSTERS;

// Barrier number `phase` (1, 2, ...) of the G CTAs sharing *counter (zero at the start of the call). The
// wait is bounded: on expiry the status is set and the counter raised past every target, whichever CTAs
// expire with this one, so that no later barrier of the call waits. False from then on.
constexpr int kBarrierGone = 1 << 30;
__device__ __forceinline__ bool tile_barrier(int* counter, int G, int phase, int* status, long long budget) {
  bool gone = false;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(counter, 1);
    const long long t0 = clock64();
    while (true) {
      int v;
      asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(counter) : "memory");
      if (v >= G * phase) {
        gone = v >= kBarrierGone;
        break;
      }
      if (clock64() - t0 > budget) {
        set_status(status, SPD_ETIMEOUT);
        atomicMax(counter, kBarrierGone);
        gone = true;
        break;
      }
    }
  }
  return !__syncthreads_or(gone);
}

// CTAs at `barriers` barriers in a row that one more CTA would have to reach (spd_selftest_tile_barrier).
__global__ void tile_barrier_probe_kernel(int* ws, int barriers, long long budget) {
  for (int i = 1; i <= barriers; ++i) tile_barrier(ws + 1, int(gridDim.x) + 1, i, ws, budget);
}

template <int KN, bool COS>
__global__ void __launch_bounds__(kGridThreads) kmeans_grid_kernel(PruneDims p, PruneWs w, int G, int res) {
  extern __shared__ __align__(16) float ksm[];
  const int K = p.K, D = p.d, m = p.m, KD = K * D;
  const int t = blockIdx.x / G, r = blockIdx.x - t * G;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int NW = kGridThreads / 32;
  float* cent = ksm;       // [K][D]
  float* rows = ksm + KD;  // res: [nl][D]
  __shared__ int8_t asg[kGridMaxRows];
  __shared__ uint16_t ord[kGridMaxRows];
  __shared__ int start[SPD_MAX_CLUSTERS + 1];
  __shared__ int idx[kGridMaxRows];
  __shared__ float av[kGridMaxRows], rinv[kGridMaxRows];
  __shared__ int cnt[SPD_MAX_CLUSTERS], ncl[SPD_MAX_CLUSTERS];
  __shared__ int changed, any_changed;
  __shared__ float seg[NW][33];
  __shared__ uint64_t rows_bar;
  const int j0 = int((long long)r * m / G), j1 = int((long long)(r + 1) * m / G), nl = j1 - j0;
  const int* ul = w.ulist + size_t(t) * m;
  const size_t row0 = size_t(t) * p.n_tok + p.off;
  const float* fin = p.feat[p.fin];
  int* meta = w.gmeta + size_t(t) * G * kGridMeta;          // [G][kGridMeta]
  float* part = w.gpart + size_t(t) * G * p.L * KD;         // [G][L][K][D] column sums of each CTA
  double* dsum = w.gdsum + size_t(t) * G * p.L * 16;        // [G][L][16] MSE / KL: sums of st1 (+ st3)
  float* gcent = w.gcent + size_t(t) * KD;                  // [K][D]
  int* bar = &w.arrive[4 * t + 2];
  int phase = 0;
  bool ok = true;  // no barrier has expired
  pdl_wait();
  for (int jj = threadIdx.x; jj < nl; jj += blockDim.x) {
    idx[jj] = ul[j0 + jj];
    av[jj] = ordered_val(w.asim[size_t(t) * p.n + ul[j0 + jj]]);
  }
  if (threadIdx.x == 0) {
    mbar_init(&rows_bar, 1);
    fence_mbar_init();
  }
  __syncthreads();
  if (res && warp == 0 && nl > 0) {
    if (lane == 0) mbar_arrive_expect_tx(&rows_bar, uint32_t(nl) * D * 4);
    __syncwarp();
    for (int jj = lane; jj < nl; jj += 32)
      bulk_load(rows + size_t(jj) * D, fin + (row0 + idx[jj]) * D, uint32_t(D) * 4, &rows_bar);
  }
  for (int e = threadIdx.x; e < KD; e += blockDim.x) {
    const int k = e / D, c = e - k * D;
    cent[e] = feat_row(p, p.fin, t, ul[int((long long)k * m / K)])[c];
  }
  if (res && nl > 0) {
    volatile int no_abort = 0;
    if (!mbar_wait(&rows_bar, 0, &no_abort, kWaitBudget)) {
      set_status(w.status, SPD_ETIMEOUT);
      mbar_wait(&rows_bar, 0, &no_abort, kWaitBudget);  // the copies land before anything reuses it
    }
  }
  auto xrow = [&](int jj) -> const float* { return res ? rows + size_t(jj) * D : fin + (row0 + idx[jj]) * D; };
  // emit(e, sum over the CTAs of src[e] of their blocks of `ld` floats) for this CTA's share of [0, n):
  // the warps sum contiguous ranges of CTAs in rank order, their sums are added in warp order
  auto reduce = [&](const float* src, size_t ld, int n, auto emit) {
    const int e0 = int((long long)r * n / G), e1 = int((long long)(r + 1) * n / G);
    for (int eb = e0; eb < e1; eb += 32) {
      const int e = eb + lane;
      float sum = 0.0f;
      if (e < e1) {
        const int c0 = warp * G / NW, c1 = (warp + 1) * G / NW;
#pragma unroll 10
        for (int cc = c0; cc < c1; ++cc) sum += __ldcg(src + cc * ld + e);
      }
      seg[warp][lane] = sum;
      __syncthreads();
      if (warp == 0 && e < e1) {
        float tot = 0.0f;
#pragma unroll
        for (int q = 0; q < NW; ++q) tot += seg[q][lane];
        emit(e, tot);
      }
      __syncthreads();
    }
  };
  for (int it = 0; it < p.iters; ++it) {
    if (threadIdx.x == 0) changed = 0;
    __syncthreads();
    assign_rows<KN>(cent, K, D, nl, it == 0, asg, &changed, xrow);
    __syncthreads();
    cluster_lists(asg, nl, K, cnt, ord, start);
    __syncthreads();
    column_sums(part + size_t(r) * p.L * KD, K, D, nl, ord, start,
                RowAccess{res ? rows : nullptr, fin, row0, idx, D, nullptr});
    __syncthreads();
    // sizes of K <= 16 clusters, the flag beside each (a reader of any cluster's sizes sees it)
    if (threadIdx.x < K) meta[r * kGridMeta + threadIdx.x] = cnt[threadIdx.x] | (changed ? 1 << 30 : 0);
    if (!(ok = tile_barrier(bar, G, ++phase, w.status, kWaitBudget))) break;
    if (threadIdx.x == 0) any_changed = 0;
    __syncthreads();
    if (warp < K) {
      int n = 0, f = 0;
      for (int cc = lane; cc < G; cc += 32) {
        const int v = __ldcg(meta + cc * kGridMeta + warp);
        n += v & ((1 << 30) - 1);
        f |= v >> 30;
      }
#pragma unroll
      for (int off = 16; off; off >>= 1) {
        n += __shfl_xor_sync(0xffffffffu, n, off);
        f |= __shfl_xor_sync(0xffffffffu, f, off);
      }
      if (lane == 0) {
        ncl[warp] = n;
        if (f) any_changed = 1;
      }
    }
    __syncthreads();
    if (it > 0 && !any_changed) break;  // the same in every CTA of the tile
    if (it + 1 == p.iters) break;       // the centroids are read by assignments only
    reduce(part, size_t(p.L) * KD, KD, [&](int e, float sum) {
      const int n = ncl[e / D];
      gcent[e] = n > 0 ? sum / float(n) : cent[e];
    });
    if (!(ok = tile_barrier(bar, G, ++phase, w.status, kWaitBudget))) break;
    for (int e = 4 * threadIdx.x; e < KD; e += 4 * blockDim.x)
      *reinterpret_cast<float4*>(cent + e) = __ldcg(reinterpret_cast<const float4*>(gcent + e));
    __syncthreads();
  }
  // the final assignment, this CTA's sums of a_j (token order) and, a layer, of the unit feature rows (raw
  // rows and st1 for the MSE and KL similarities). The loop left right after a barrier, without a reduction
  // behind it: no CTA still reads the blocks written here.
  for (int jj = threadIdx.x; jj < nl; jj += blockDim.x) w.assign[size_t(t) * m + j0 + jj] = asg[jj];
  if (threadIdx.x < K) {
    float a = 0.0f;
    for (int j = start[threadIdx.x]; j < start[threadIdx.x + 1]; ++j) a += av[ord[j]];
    meta[r * kGridMeta + SPD_MAX_CLUSTERS + threadIdx.x] = __float_as_int(a);
  }
  for (int l = 0; l < p.L; ++l) {
    const float* rstat = (COS ? w.inv : w.st1) + (size_t(l) * p.n_tiles + t) * p.n;
    __syncthreads();  // the previous layer's statistics are no longer read
    for (int jj = threadIdx.x; jj < nl; jj += blockDim.x) rinv[jj] = rstat[idx[jj]];
    __syncthreads();
    if (!COS && threadIdx.x < K) {  // token order, fp64 (KL: the fp64 log-sum-exps)
      const float* lo = p.sim == SPD_SIM_KL ? w.st3 + (size_t(l) * p.n_tiles + t) * p.n : nullptr;
      double a = 0.0;
      for (int jj = 0; jj < nl; ++jj)
        if (asg[jj] == int(threadIdx.x)) a += double(rinv[jj]) + (lo ? double(lo[idx[jj]]) : 0.0);
      dsum[(size_t(r) * p.L + l) * 16 + threadIdx.x] = a;
    }
    column_sums(part + (size_t(r) * p.L + l) * KD, K, D, nl, ord, start,
                RowAccess{res && l == p.fin ? rows : nullptr, p.feat[l], row0, idx, D,
                          COS ? rinv : static_cast<float*>(nullptr)});
  }
  ok = tile_barrier(bar, G, ++phase, w.status, kWaitBudget) && ok;
  pdl_launch_dependents();
  reduce(part, size_t(p.L) * KD, p.L * KD, [&](int e, float sum) { w.csum[size_t(t) * p.L * KD + e] = sum; });
  if (r != 0) return;
  if (!ok) {  // an expired barrier (the status tells): the sizes may be anything, and nothing is selected by them
    if (threadIdx.x < SPD_MAX_CLUSTERS) ncl[threadIdx.x] = 0;
    __syncthreads();
  }
  if (warp < K) {  // lane sums over CTAs lane, lane + 32, ..., then a butterfly: a fixed order
    float a = 0.0f;
    for (int cc = lane; cc < G; cc += 32) a += __int_as_float(__ldcg(meta + cc * kGridMeta + SPD_MAX_CLUSTERS + warp));
    a = warp_sum(a);
    if (lane == 0) {
      w.counts[t * 16 + warp] = ncl[warp];
      w.asum[t * 16 + warp] = a;
    }
    if (!COS)
      for (int l = 0; l < p.L; ++l) {
        double d = 0.0;
        for (int cc = lane; cc < G; cc += 32) d += __ldcg(dsum + (size_t(cc) * p.L + l) * 16 + warp);
        d = warp_sum_d(d);
        if (lane == 0) w.ssum[(size_t(t) * p.L + l) * 16 + warp] = d;
      }
  }
  if (warp == 0) warp_quotas(ncl, K, p.n_cmp, w.quotas + t * 16);
}

// ---- 4c. K-means of many tiles: one sweep over the rows an iteration ------------------------------
// K = 4. A cluster of KC CTAs per tile, one CTA an SM, as many as the tiles leave (64 tiles: 2). The rows
// of all tiles exceed L2 (531 x 4 KB a LLaVA tile), so what counts is how often they are read and how many
// bytes are in flight: every thread copies its four columns of 16 rows at a time (8 where rows are wider
// than 1024) with 16-byte asynchronous copies into a ring of such steps, and one sweep does the
// assignment of a step's rows (two a warp) and then their column sums from shared memory, four columns a
// thread in registers. (One bulk copy a row held the whole kernel at 2.5 TB/s: 165 us.) From the second sweep on
// it also adds the unit rows, which are the final layer's cluster sums if the assignment repeats. Every second
// sweep runs backwards: the rows that the last one read end up in L2. So a tile whose assignment repeats at once
// is read twice for K-means and once a further layer, where 4 CTAs a tile re-reading the rows through registers read
// it five times: 64 tiles 234 -> 156 us serialised, of which the copies alone take 76; the assignment (with
// the centroids in registers up to 1024 columns) and the sums are chains of shared-memory loads of 8 warps.
constexpr int kStreamThreads = 256;
constexpr size_t kStreamSmem = 226 * 1024;  // dynamic shared memory of a CTA
// Column groups of a thread (rows of up to 1024 or 2048 floats) and rows of a step.
__host__ __device__ inline int stream_groups(int D) { return D <= 4 * kStreamThreads ? 1 : 2; }
__host__ __device__ constexpr int stream_step(int CG) { return CG == 1 ? 16 : 8; }
// Bytes of the arrays before the ring, and the steps that then fit.
__host__ __device__ inline size_t stream_head(int D, int nl_max) {
  return (size_t(8) * D * sizeof(float) + size_t(nl_max) * 7 + 15) / 16 * 16;
}
inline int stream_slots(int D, int nl_max, size_t smem) {
  const size_t head = stream_head(D, nl_max), slot = size_t(stream_step(stream_groups(D))) * D * sizeof(float);
  return head >= smem ? 0 : int((smem - head) / slot);
}

// 16 bytes from global to shared memory, past L1; groups of them complete in the order of their commits.
__device__ __forceinline__ void copy_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copy_async_wait() {  // all but the thread's last N groups have landed
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

template <int KC, int CG, bool COS>
__global__ void __launch_bounds__(kStreamThreads, 1) kmeans_stream_kernel(PruneDims p, PruneWs w, int slots) {
  extern __shared__ __align__(16) float ksm[];
  constexpr int K = 4, SR = stream_step(CG), SB = 8 / CG;  // rows a step, rows in flight in the sums
  const int D = p.d, m = p.m;
  const int nl_max = (m + KC - 1) / KC;
  float* cent = ksm;            // [K][D]
  float* part = cent + K * D;   // [K][D]
  float* rinv = part + K * D;   // [nl_max] scale (cosine) or st1 (MSE, KL) of the current layer
  uint16_t* idx = reinterpret_cast<uint16_t*>(rinv + nl_max);
  int8_t* asg = reinterpret_cast<int8_t*>(idx + nl_max);
  float* ring = ksm + stream_head(D, nl_max) / sizeof(float);  // [slots][SR][D]
  // during a sweep, in part's place (4 D >= 2 SR kStreamThreads / 32 floats): each warp's list of a step's rows by
  // cluster, as offsets into the step, and their scales
  int* ord_off = reinterpret_cast<int*>(part) + (threadIdx.x >> 5) * SR;
  float* ord_scale = part + (kStreamThreads / 32 + (threadIdx.x >> 5)) * SR;
  __shared__ int cnt[SPD_MAX_CLUSTERS], ncl[SPD_MAX_CLUSTERS];
  __shared__ int changed, any_changed;
  __shared__ float asum_part[K];
  __shared__ double ssum_part[K];
  cg::cluster_group cl = cg::this_cluster();
  const int rank = int(cl.block_rank());
  const int t = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int j0 = rank * m / KC, j1 = (rank + 1) * m / KC, nl = j1 - j0;
  const int* ul = w.ulist + size_t(t) * m;
  const size_t row0 = size_t(t) * p.n_tok + p.off;
  const float* fin = p.feat[p.fin];
  pdl_launch_dependents();
  pdl_wait();
  const float* frin = w.inv + (size_t(p.fin) * p.n_tiles + t) * p.n;
  for (int jj = threadIdx.x; jj < nl; jj += blockDim.x) {
    const int i = ul[j0 + jj];
    idx[jj] = uint16_t(i);
    if (COS) rinv[jj] = frin[i];
  }
  __syncthreads();
  const int ns = (nl + SR - 1) / SR;  // steps of a sweep
  // copies step i of a sweep over layer rows f into slot i % slots (one group, empty past the end)
  auto issue = [&](const float* f, int i, bool back) {
    if (i < ns) {
      const int r0 = (back ? ns - 1 - i : i) * SR, rows = min(SR, nl - r0);
      float* dst = ring + size_t(i % slots) * SR * D;
#pragma unroll 4
      for (int v = 0; v < rows; ++v) {
        const float* src = f + (row0 + idx[r0 + v]) * D;
#pragma unroll
        for (int q = 0; q < CG; ++q) {
          const int c = 4 * (threadIdx.x + kStreamThreads * q);
          if (c < D) copy_async16(dst + size_t(v) * D + c, src + c);
        }
      }
    }
    copy_async_commit();
  };
  auto start = [&](const float* f, bool back) {  // the first two steps of a sweep
    issue(f, 0, back);
    issue(f, 1, back);
  };
  ulonglong2 acc[K][CG], unit[K][CG];  // four columns each, as two packed pairs
  // one sweep: assignment (where `assign`) and column sums of the rows (acc, where `raw`) and of the rows times
  // rinv (unit, where `units`); its first two steps were issued by start()
  auto sweep = [&](const float* f, bool back, bool assign, bool first, bool raw, bool units) {
#pragma unroll
    for (int k = 0; k < K; ++k)
#pragma unroll
      for (int q = 0; q < CG; ++q) acc[k][q] = unit[k][q] = make_ulonglong2(0, 0);
    ulonglong2 cr[CG == 1 ? 4 : 1][CG == 1 ? 8 : 1];  // centroids of rows of up to 1024 floats
    if (CG == 1 && assign) {
#pragma unroll
      for (int k = 0; k < (CG == 1 ? 4 : 1); ++k)
#pragma unroll
        for (int j = 0; j < (CG == 1 ? 8 : 1); ++j) {
          const int c = 4 * lane + 128 * j;
          cr[k][j] = c < D ? *reinterpret_cast<const ulonglong2*>(cent + k * D + c) : make_ulonglong2(0, 0);
        }
    }
    for (int i = 0; i < ns; ++i) {
      // with three slots the step after the next is issued before this one is used, with two after it
      if (slots > 2) issue(f, i + 2, back);
      if (slots > 2) copy_async_wait<2>();
      else copy_async_wait<1>();
      __syncthreads();  // every thread's columns of step i have landed
      const int r0 = (back ? ns - 1 - i : i) * SR, rows = min(SR, nl - r0);
      const float* base = ring + size_t(i % slots) * SR * D;
      if (assign) {
        constexpr int RP = SR / 8;  // rows a warp
        const int v0 = warp * RP;
        auto row = [&](int q) { return base + size_t(v0 + q) * D; };
        if (v0 < rows) {
          if constexpr (CG == 1) assign4_regs<RP>(cr, D, rows - v0, first, asg + r0 + v0, &changed, row);
          else assign4_rows<RP>(cent, D, rows - v0, first, asg + r0 + v0, &changed, row);
        }
        __syncthreads();
      }
      // the step's rows by cluster, in token order within each (every warp for itself): a row then costs its
      // load and two packed additions a pair set
      const int a = lane < rows ? asg[r0 + lane] : K;
      int first_of[K + 1], rank_of = 0;
      first_of[0] = 0;
#pragma unroll
      for (int k = 0; k < K; ++k) {
        const uint32_t who = __ballot_sync(0xffffffffu, a == k);
        if (a == k) rank_of = first_of[k] + __popc(who & ((1u << lane) - 1));
        first_of[k + 1] = first_of[k] + __popc(who);
      }
      if (lane < rows) {
        ord_off[rank_of] = lane * D;
        if (units) ord_scale[rank_of] = rinv[r0 + lane];
      }
      __syncwarp();
#pragma unroll
      for (int k = 0; k < K; ++k)
        for (int v = first_of[k]; v < first_of[k + 1]; v += SB) {
          ulonglong2 x[SB][CG];
#pragma unroll
          for (int e = 0; e < SB; ++e)
#pragma unroll
            for (int q = 0; q < CG; ++q) {
              const int c = 4 * (threadIdx.x + kStreamThreads * q);
              x[e][q] = v + e < first_of[k + 1] && c < D
                            ? *reinterpret_cast<const ulonglong2*>(base + ord_off[v + e] + c)
                            : make_ulonglong2(0, 0);
            }
          if (raw)
#pragma unroll
            for (int e = 0; e < SB; ++e)
#pragma unroll
              for (int q = 0; q < CG; ++q) {
                acc[k][q].x = add_f32x2(acc[k][q].x, x[e][q].x);
                acc[k][q].y = add_f32x2(acc[k][q].y, x[e][q].y);
              }
          if (units)
#pragma unroll
            for (int e = 0; e < SB; ++e) {
              const uint32_t sb = v + e < first_of[k + 1] ? __float_as_uint(ord_scale[v + e]) : 0u;
              const uint64_t sc = uint64_t(sb) << 32 | sb;
#pragma unroll
              for (int q = 0; q < CG; ++q) {
                unit[k][q].x = fma_f32x2(x[e][q].x, sc, unit[k][q].x);
                unit[k][q].y = fma_f32x2(x[e][q].y, sc, unit[k][q].y);
              }
            }
        }
      __syncthreads();  // the step's slot may be refilled
      if (slots <= 2) issue(f, i + 2, back);
    }
    copy_async_wait<0>();  // (empty groups past the end)
  };
  auto to_part = [&](const ulonglong2 (&v)[K][CG]) {
#pragma unroll
    for (int k = 0; k < K; ++k)
#pragma unroll
      for (int q = 0; q < CG; ++q) {
        const int c = 4 * threadIdx.x + 4 * kStreamThreads * q;
        if (c < D) *reinterpret_cast<ulonglong2*>(part + k * D + c) = v[k][q];
      }
  };
  start(fin, false);
  for (int e = 4 * threadIdx.x; e < K * D; e += 4 * blockDim.x) {
    const int k = e / D, c = e - k * D;
    *reinterpret_cast<float4*>(cent + e) = *reinterpret_cast<const float4*>(feat_row(p, p.fin, t, ul[(k * m) / K]) + c);
  }
  bool done = false;  // the last sweep's unit sums are the final layer's cluster sums
  for (int it = 0; it < p.iters; ++it) {
    const bool units = COS && (it > 0 || it + 1 == p.iters);
    if (threadIdx.x == 0) changed = 0;
    if (threadIdx.x < SPD_MAX_CLUSTERS) cnt[threadIdx.x] = 0;
    __syncthreads();
    sweep(fin, it & 1, true, it == 0, true, units);
    for (int jj = threadIdx.x; jj < nl; jj += blockDim.x) atomicAdd(&cnt[asg[jj]], 1);
    to_part(acc);
    cl.sync();
    if (warp == 0) {
      const int f = lane < KC ? *cl.map_shared_rank(&changed, lane) : 0;
      const int any = __any_sync(0xffffffffu, f != 0);
      for (int k = 0; k < K; ++k) {
        int n = lane < KC ? cl.map_shared_rank(cnt, lane)[k] : 0;
#pragma unroll
        for (int off = 16; off; off >>= 1) n += __shfl_xor_sync(0xffffffffu, n, off);
        if (lane == 0) ncl[k] = n;
      }
      if (lane == 0) any_changed = any;
    }
    __syncthreads();
    done = (it > 0 && !any_changed) || it + 1 == p.iters;  // the same in every CTA of the cluster
    if (done) break;
    start(fin, (it + 1) & 1);
    cluster_column_reduce<KC>(cl, part, K, D, rank, [&](int k, int c, float4 v) {
      const float n = float(ncl[k]);
      if (n > 0.0f) v = make_float4(v.x / n, v.y / n, v.z / n, v.w / n);
      else v = *reinterpret_cast<const float4*>(cent + k * D + c);
      for (int rr = 0; rr < KC; ++rr) *reinterpret_cast<float4*>(cl.map_shared_rank(cent, rr) + k * D + c) = v;
    });
    cl.sync();
  }
  // the layers, the final one first (its sums are there): the next one's rows are on their way meanwhile
  const int last = p.L == 1 ? p.fin : (p.fin == p.L - 1 ? p.L - 2 : p.L - 1);
  auto layer = [&](int li) { return li == 0 ? p.fin : (li <= p.fin ? li - 1 : li); };
  if (p.L > 1) start(p.feat[layer(1)], false);
  for (int jj = threadIdx.x; jj < nl; jj += blockDim.x) w.assign[size_t(t) * m + j0 + jj] = asg[jj];
  if (threadIdx.x < 32 * K) {  // a warp a cluster: its a_j, lanes' shares in token order, then a butterfly
    float a = 0.0f;
    for (int jj = lane; jj < nl; jj += 32)
      if (asg[jj] == warp) a += ordered_val(w.asim[size_t(t) * p.n + idx[jj]]);
    a = warp_sum(a);
    if (lane == 0) asum_part[warp] = a;
  }
  for (int li = 0; li < p.L; ++li) {
    const int l = layer(li);
    const float* rstat = (COS ? w.inv : w.st1) + (size_t(l) * p.n_tiles + t) * p.n;
    if (li > 0 || !COS) {
      __syncthreads();
      for (int jj = threadIdx.x; jj < nl; jj += blockDim.x) rinv[jj] = rstat[idx[jj]];
      __syncthreads();
    }
    if (!COS && threadIdx.x == 0) {  // token order, fp64 (KL: the fp64 log-sum-exps)
      const float* lo = p.sim == SPD_SIM_KL ? w.st3 + (size_t(l) * p.n_tiles + t) * p.n : nullptr;
      for (int k = 0; k < K; ++k) ssum_part[k] = 0.0;
      for (int jj = 0; jj < nl; ++jj)
        ssum_part[asg[jj]] += double(rinv[jj]) + (lo ? double(lo[idx[jj]]) : 0.0);
    }
    if (li > 0) {
      sweep(p.feat[l], false, false, false, !COS, COS);
      if (li + 1 < p.L) start(p.feat[layer(li + 1)], false);
    }
    // (no peer reads the sums of the last iteration, which the loop left before its reduction)
    if (COS) to_part(unit);
    else to_part(acc);
    cl.sync();
    float* csum = w.csum + (size_t(t) * p.L + l) * K * D;
    cluster_column_reduce<KC>(cl, part, K, D, rank, [&](int k, int c, float4 sum) {
      *reinterpret_cast<float4*>(csum + k * D + c) = sum;
    });
    if (!COS && rank == 0 && warp == 1) {  // CTA sums added in rank order
      for (int k = 0; k < K; ++k) {
        const double sr = lane < KC ? cl.map_shared_rank(ssum_part, lane)[k] : 0.0;
        double a = 0.0;
        for (int rr = 0; rr < KC; ++rr) a += __shfl_sync(0xffffffffu, sr, rr);
        if (lane == 0) w.ssum[(size_t(t) * p.L + l) * 16 + k] = a;
      }
    }
    if (l == last && rank == 0 && warp == 0) {
      for (int k = 0; k < K; ++k) {
        const float ar = lane < KC ? cl.map_shared_rank(asum_part, lane)[k] : 0.0f;
        float a = 0.0f;
        for (int rr = 0; rr < KC; ++rr) a += __shfl_sync(0xffffffffu, ar, rr);
        if (lane == 0) {
          w.counts[t * 16 + k] = ncl[k];
          w.asum[t * 16 + k] = a;
        }
      }
      warp_quotas(ncl, K, p.n_cmp, w.quotas + t * 16);
    }
    cl.sync();  // the peers' shared memory is read above
  }
}

// ---- 6. per-token Eq. 3 scores ----------------------------------------------------------------
// Per layer, with X_k the cluster's column sums and c = |C_k|, the sum over the other members j:
//   cos: sum_j f_i.f_j = f_i.(X_k - f_i)                                     (f = F / |F|)
//   MSE: sum_j -|F_i - F_j|^2 / d = -[(c - 1) |F_i|^2 - 2 F_i.(X_k - F_i) + (Q_k - |F_i|^2)] / d
//   KL:  sum_j -KL(P_i || P_j) = -c sum_c P_i,c (log P_i,c - (X_k,c - S_k) / c)
//        (the j = i term is 0; (X_k - S_k) / c is the cluster mean of log P_j, so every product
//        is of a probability and an O(1) difference of logs, with no cancellation of large sums)
// (Q_k, S_k: the cluster's sums of |F_j|^2 and of lse_j.)
// One warp per token. The cosine instance is held to 80 registers so that three CTAs share an SM
// (a few bytes of spills; 64 tiles about 10 us faster than at 97 registers and two CTAs).
template <int SIM>
__global__ void __launch_bounds__(256, SIM == SPD_SIM_COS ? 3 : 1) score_kernel(PruneDims p, PruneWs w) {
  pdl_launch_dependents();
  pdl_wait();
  const int t = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int j = blockIdx.x * 8 + warp;
  if (j >= p.m) return;
  const int i = w.ulist[size_t(t) * p.m + j];
  const int k = w.assign[size_t(t) * p.m + j];
  const int cnt = w.counts[t * 16 + k];
  const float ai = ordered_val(w.asim[size_t(t) * p.n + i]);
  float s;
  if (cnt <= 1) {
    s = p.wa * 2.0f * ai;
  } else {
    float acc = 0.0f;
    for (int l = 0; l < p.L; ++l) {
      const float wl = (l == p.fin) ? p.wf : p.w[l];
      if (wl == 0.0f) continue;
      const float4* x4 = reinterpret_cast<const float4*>(feat_row(p, l, t, i));
      const size_t so = (size_t(l) * p.n_tiles + t) * p.n + i;
      const float iv = SIM == SPD_SIM_COS ? w.inv[so] : 1.0f;
      // KL in fp64: log P_i,c = x_c - lse_i and the cluster mean of log P_j,c
      const double lse = SIM == SPD_SIM_KL ? double(w.st1[so]) + double(w.st3[so]) : 0.0;
      const double sbar = SIM == SPD_SIM_KL ? w.ssum[(size_t(t) * p.L + l) * 16 + k] / double(cnt) : 0.0;
      const float4* c4 =
          reinterpret_cast<const float4*>(w.csum + ((size_t(t) * p.L + l) * p.K + k) * p.d);
      // 16-byte loads, sixteen in flight per lane, two independent chains
      const int d4 = p.d / 4;
      float dot0 = 0.0f, dot1 = 0.0f;
      double kdot = 0.0;  // KL
      for (int cb = lane; cb < d4; cb += 256) {
        float4 xv[8], cv[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int c = cb + 32 * u;
          xv[u] = c < d4 ? x4[c] : make_float4(0.f, 0.f, 0.f, 0.f);
          cv[u] = c < d4 ? c4[c] : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          // cos: f.(X - f) with f = x |x|^-1; MSE: x.(X - x); KL: P.(log P - mean_j log P_j)
          const float b0 = xv[u].x * iv, b1 = xv[u].y * iv, b2 = xv[u].z * iv, b3 = xv[u].w * iv;
          if constexpr (SIM == SPD_SIM_KL) {
            if (cb + 32 * u >= d4) continue;  // a zero-filled slot is no zero term here
            const double dn = double(cnt);
            const double l0 = double(b0) - lse, l1 = double(b1) - lse, l2 = double(b2) - lse,
                         l3 = double(b3) - lse;
            kdot += exp(l0) * (l0 - (double(cv[u].x) / dn - sbar)) +
                    exp(l1) * (l1 - (double(cv[u].y) / dn - sbar)) +
                    exp(l2) * (l2 - (double(cv[u].z) / dn - sbar)) +
                    exp(l3) * (l3 - (double(cv[u].w) / dn - sbar));
          } else {
            const float part =
                b0 * (cv[u].x - b0) + b1 * (cv[u].y - b1) + b2 * (cv[u].z - b2) + b3 * (cv[u].w - b3);
            if (u & 1) dot1 += part;
            else dot0 += part;
          }
        }
      }
      const float dot = warp_sum(dot0 + dot1);
      float term = dot;
      if (SIM == SPD_SIM_MSE) {
        const float sk = float(w.ssum[(size_t(t) * p.L + l) * 16 + k]), st = w.st1[so];
        term = -(float(cnt - 1) * st - 2.0f * dot + (sk - st)) / float(p.d);
      } else if (SIM == SPD_SIM_KL) {
        term = float(-double(cnt) * warp_sum_d(kdot));
      }
      acc += wl * term;
    }
    const float inv_c = 1.0f / float(cnt - 1);
    s = acc * inv_c + p.wa * (ai + (w.asum[t * 16 + k] - ai) * inv_c);
  }
  if (lane == 0) w.score[size_t(t) * p.m + j] = s;
}

// ---- received attention from full maps (Sec. 4.1.1 without [CLS]) ------------------------------
// Column sums of attention maps: CTA (column block, map, row split) adds rows [q0, q1) of its 1024
// columns (thread: four adjacent columns, float4 loads, eight rows in flight) in row order.
__global__ void __launch_bounds__(256) received_colsum_kernel(const float* maps, int n_q,
                                                              int n_k, int rows_per_split,
                                                              float* __restrict__ partial) {
  pdl_launch_dependents();
  pdl_wait();
  const int c4 = blockIdx.x * 256 + threadIdx.x;  // float4 column group
  const int mp = blockIdx.y, sp = blockIdx.z, n_maps = gridDim.y;
  if (4 * c4 >= n_k) return;
  const int q0 = sp * rows_per_split, q1 = min(n_q, q0 + rows_per_split);
  const float4* src = reinterpret_cast<const float4*>(maps + size_t(mp) * n_q * n_k) + c4;
  const size_t ld4 = n_k / 4;
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int q = q0; q < q1; q += 8) {
    float4 v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u)
      v[u] = q + u < q1 ? __ldcs(src + size_t(q + u) * ld4) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      acc.x += v[u].x;
      acc.y += v[u].y;
      acc.z += v[u].z;
      acc.w += v[u].w;
    }
  }
  reinterpret_cast<float4*>(partial + (size_t(sp) * n_maps + mp) * n_k)[c4] = acc;
}

// out[m][j] = sum over the members i of group j (ascending) of (sum over splits, in order, of the
// partial column sums) / n_q; without groups j = i.
__global__ void __launch_bounds__(256) received_finish_kernel(const float* partial,
                                                              int n_maps, int n_k, int n_splits,
                                                              float inv_nq,
                                                              const int32_t* gstart,
                                                              const int32_t* gmem,
                                                              int n_out, float* __restrict__ out,
                                                              int* status) {
  pdl_launch_dependents();
  pdl_wait();
  const int j = blockIdx.x * 256 + threadIdx.x, mp = blockIdx.y;
  if (j >= n_out) return;
  auto col = [&](int i) {
    float s = 0.0f;
    for (int sp = 0; sp < n_splits; ++sp) s += partial[(size_t(sp) * n_maps + mp) * n_k + i];
    return s * inv_nq;
  };
  float v = 0.0f;
  if (gstart) {
    for (int e = gstart[j]; e < gstart[j + 1]; ++e) {
      const int i = gmem[e];
      if (i < 0 || i >= n_k) {
        set_status(status, SPD_EINVAL);
        continue;
      }
      v += col(i);
    }
  } else {
    v = col(j);
  }
  out[size_t(mp) * n_out + j] = v;
}

// ---- 7. per-cluster bottom-N_k, compaction, outputs -------------------------------------------
__global__ void __launch_bounds__(kRankThreads) select_kernel(PruneDims p, PruneWs w, int32_t* keep_idx,
                                                              uint8_t* kind, int8_t* cluster, float* scores) {
  pdl_launch_dependents();
  pdl_wait();
  __shared__ __align__(16) uint64_t keys[4096];  // (cluster, score) of the non-anchor list
  __shared__ int rank[kRankThreads];
  __shared__ uint8_t kept[4096];
  __shared__ int tmp[32];
  __shared__ int seg[SPD_MAX_CLUSTERS + 1];
  __shared__ int quota[SPD_MAX_CLUSTERS];
  const int t = blockIdx.y, nb = gridDim.x, m = p.m;
  const int* ul = w.ulist + size_t(t) * m;
  int8_t* role = w.role + size_t(t) * p.n;
  for (int j = threadIdx.x; j < ((m + 1) & ~1); j += blockDim.x)
    keys[j] = j < m ? (uint64_t(w.assign[size_t(t) * m + j]) << 32) | ordered_key(w.score[size_t(t) * m + j])
                    : ~0ull;
  if (nb == 1)
    for (int i = threadIdx.x; i < p.n; i += blockDim.x) kept[i] = uint8_t(role[i]);
  if (threadIdx.x == 0) {
    int acc = 0;
    for (int k = 0; k < p.K; ++k) {
      seg[k] = acc;
      acc += w.counts[t * 16 + k];
      quota[k] = w.quotas[t * 16 + k];
    }
    seg[p.K] = acc;
  }
  __syncthreads();
  const int j0 = blockIdx.x * m / nb, j1 = (blockIdx.x + 1) * m / nb;
  if (j0 < j1) {  // m > 0 (block-uniform)
    count_ranks(keys, m, j0, j1, rank);
    __syncthreads();
    // the key at sorted position r of cluster k's segment is kept iff r - seg[k] < quota[k]
    for (int j = j0 + threadIdx.x; j < j1; j += blockDim.x) {
      const int k = int(keys[j] >> 32);
      if (rank[j - j0] - seg[k] < quota[k]) {
        if (nb == 1) kept[ul[j]] = 2;
        else role[ul[j]] = 2;  // the anchors' flags are 1
      }
    }
  }
  if (!last_cta(&w.arrive[4 * t + 1], nb)) return;
  if (nb > 1)
    for (int i = threadIdx.x; i < p.n; i += blockDim.x) kept[i] = uint8_t(__ldcg(role + i));
  __syncthreads();
  const int base = threadIdx.x * 4;
  int nk = 0;
  for (int q = 0; q < 4; ++q)
    if (base + q < p.n) nk += kept[base + q] != 0;
  int pos = block_scan_excl(nk, tmp, nullptr);
  for (int q = 0; q < 4; ++q) {
    const int i = base + q;
    if (i >= p.n) break;
    if (kept[i]) {
      if (pos < p.keep) keep_idx[size_t(t) * p.keep + pos] = i;
      else set_status(w.status, SPD_EINVAL);
      ++pos;
    }
    if (kind) kind[size_t(t) * p.n + i] = kept[i];
    if (kept[i] == 1) {
      if (cluster) cluster[size_t(t) * p.n + i] = -1;
      if (scores) scores[size_t(t) * p.n + i] = INFINITY;
    }
  }
  for (int j = threadIdx.x; j < m; j += blockDim.x) {
    if (cluster) cluster[size_t(t) * p.n + ul[j]] = int8_t(w.assign[size_t(t) * m + j]);
    if (scores) scores[size_t(t) * p.n + ul[j]] = w.score[size_t(t) * m + j];
  }
}

__global__ void gather_bf16_kernel(const float* src, int n_tok, int d, int off, const int32_t* idx,
                                   int keep,
                                   __nv_bfloat16* __restrict__ dst, int* status) {
  pdl_launch_dependents();
  pdl_wait();
  const int j = blockIdx.x, t = blockIdx.y;
  const int i = idx[size_t(t) * keep + j];
  if (i < 0 || i >= n_tok - off) {
    if (threadIdx.x == 0) set_status(status, SPD_EINVAL);
    return;
  }
  const float4* s = reinterpret_cast<const float4*>(src + (size_t(t) * n_tok + off + i) * d);
  uint2* o = reinterpret_cast<uint2*>(dst + (size_t(t) * keep + j) * d);
  for (int c = threadIdx.x; c < d / 4; c += blockDim.x) {
    const float4 v = s[c];
    __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
    o[c] = make_uint2(*reinterpret_cast<uint32_t*>(&lo), *reinterpret_cast<uint32_t*>(&hi));
  }
}

int validate(const spd_prune_cfg* c, PruneDims* p) {
  if (!c) return fail(SPD_EINVAL, "null prune config");
  if (c->n_tiles < 1 || c->n_layers < 1 || c->n_layers > SPD_MAX_FEAT_LAYERS)
    return fail(SPD_EINVAL, "n_tiles >= 1 and n_layers in [1, %d] required", SPD_MAX_FEAT_LAYERS);
  if (c->final_layer < 0 || c->final_layer >= c->n_layers) return fail(SPD_EINVAL, "bad final_layer");
  const int off = c->has_cls ? 1 : 0;
  const int n = c->n_tok - off;
  if (n < 1 || n > 4096) return fail(SPD_EINVAL, "patch count must lie in [1, 4096]");
  if (c->d_feat < 4 || c->d_feat % 4 || c->d_feat > 4096)
    return fail(SPD_EINVAL, "d_feat must be a multiple of 4 in [4, 4096]");
  if (c->n_heads < 1) return fail(SPD_EINVAL, "n_heads >= 1 required");
  if (c->attn_form != 0 && c->attn_form != 1) return fail(SPD_EINVAL, "attn_form must be 0 or 1");
  if (c->attn_form == 0 && !c->has_cls) return fail(SPD_EINVAL, "CLS-row attention needs has_cls");
  if (c->keep < 1 || c->keep > n) return fail(SPD_EINVAL, "keep must lie in [1, n_patch]");
  if (c->n_clusters < 1 || c->n_clusters > SPD_MAX_CLUSTERS) return fail(SPD_EINVAL, "bad n_clusters");
  if (size_t(c->n_clusters) * c->d_feat > 24576)
    return fail(SPD_EINVAL, "n_clusters * d_feat must not exceed 24576");
  if (c->kmeans_iters < 1) return fail(SPD_EINVAL, "kmeans_iters >= 1 required");
  if (!(c->anchor_ratio >= 0.0 && c->anchor_ratio <= 1.0))
    return fail(SPD_EINVAL, "anchor_ratio must lie in [0, 1]");
  if (c->sim_kind < SPD_SIM_COS || c->sim_kind > SPD_SIM_KL) return fail(SPD_EINVAL, "bad sim_kind");
  if (c->ablate & ~(SPD_PRUNE_NO_FINAL_SIM | SPD_PRUNE_NO_ANCHOR_SIM))
    return fail(SPD_EINVAL, "unknown ablate bits");
  p->sim = c->sim_kind;
  p->wf = (c->ablate & SPD_PRUNE_NO_FINAL_SIM) ? 0.0f : 1.0f;
  p->wa = (c->ablate & SPD_PRUNE_NO_ANCHOR_SIM) ? 0.0f : 1.0f;
  p->n_tiles = c->n_tiles;
  p->n_tok = c->n_tok;
  p->off = off;
  p->n = n;
  p->d = c->d_feat;
  p->L = c->n_layers;
  p->fin = c->final_layer;
  p->H = c->n_heads;
  p->form = c->attn_form;
  p->n_att = c->attn_form == 0 ? c->n_tok : n;
  p->keep = c->keep;
  p->K = c->n_clusters;
  p->iters = c->kmeans_iters;
  p->n_anc = int(floor(double(c->keep) * c->anchor_ratio + 0.5));
  if (p->n_anc > c->keep) p->n_anc = c->keep;
  p->n_cmp = c->keep - p->n_anc;
  p->m = n - p->n_anc;
  for (int l = 0; l < SPD_MAX_FEAT_LAYERS; ++l) {
    p->w[l] = c->layer_weight[l];
    p->feat[l] = nullptr;
  }
  return SPD_OK;
}

// Dynamic shared memory of the resident K-means: its limit, and what p takes (a CTA's rows, centroids and sums).
constexpr size_t kResSmem = 200 * 1024;
size_t res_bytes(const PruneDims& p) {
  return (size_t((p.m + 15) / 16) + 2 * size_t(p.K)) * p.d * sizeof(float);
}
// Whether a call may be one of the few, large tiles that K-means spreads over the whole GPU (prune_plan
// decides with what the device holds): workspace is set aside for these alone. The others' rows are resident in
// clusters, of which 152 SMs hold kResTiles at once.
constexpr int kResTiles = 7;
bool grid_tile(const PruneDims& p) {
  return p.n_tiles <= 10 && p.m > 0 && (res_bytes(p) > kResSmem || p.n_tiles > kResTiles);
}
// Most CTAs a tile of that form.
int grid_ctas(const PruneDims& p) { return std::min(kGridMaxCtas / p.n_tiles, (p.m + 3) / 4); }

PruneWs carve(const PruneDims& p, Carve& cv) {
  PruneWs w;
  const size_t T = p.n_tiles;
  w.status = cv.status();
  w.a_v = cv.take<float>(T * p.n);
  w.inv = cv.take<float>(T * p.n * p.L);
  const size_t nst = p.sim == SPD_SIM_COS ? 0 : T * p.n * p.L;
  w.st1 = cv.take<float>(nst);
  w.st2 = cv.take<float>(p.sim == SPD_SIM_KL ? nst : 0);
  w.st3 = cv.take<float>(p.sim == SPD_SIM_KL ? nst : 0);
  w.role = cv.take<int8_t>(T * p.n);
  w.alist = cv.take<int32_t>(T * (p.n_anc + 1));
  w.ulist = cv.take<int32_t>(T * (p.m + 1));
  w.asim = cv.take<uint32_t>(T * p.n);
  w.assign = cv.take<int32_t>(T * (p.m + 1));
  w.counts = cv.take<int32_t>(T * 16);
  w.quotas = cv.take<int32_t>(T * 16);
  w.asum = cv.take<float>(T * 16);
  w.csum = cv.take<float>(T * p.L * p.K * p.d);
  w.ssum = cv.take<double>(T * p.L * 16);
  w.score = cv.take<float>(T * (p.m + 1));
  w.arrive = cv.take<int>(T * 4);
  const size_t gc = grid_tile(p) ? T * grid_ctas(p) : 0;  // CTAs of all tiles
  w.gpart = cv.take<float>(gc * p.L * p.K * p.d);
  w.gcent = cv.take<float>(gc ? T * p.K * p.d : 0);
  w.gdsum = cv.take<double>(gc * p.L * 16);
  w.gmeta = cv.take<int>(gc * kGridMeta);
  return w;
}

// Shared-memory carveout of the kernels around K-means, in percent: with the driver's choice fewer CTAs of
// anchor_sim_kernel share an SM than its registers allow (64 tiles, us a call: 446 with the driver's choice,
// 409 / 412 / 415 / 446 at 25 / 50 / 75 / 100 %; one tile 75, 68 / 66 / 71 / 72).
constexpr int kPruneCarveout = 50;
int g_res_clusters = -1;                 // 16-CTA clusters of it the GPU holds at once
int g_stream_clusters[9] = {};           // KC-CTA clusters of the one-sweep form, by KC
bool g_grid_fits = false;                // one CTA an SM of the whole-GPU form can be resident

template <int KC, bool RES, int KN, bool FUSED = false>
cudaError_t launch_kmeans(const PruneDims& p, const PruneWs& w, const PruneOut& out, size_t smem,
                          cudaStream_t st) {
  auto kern = FUSED ? kmeans_kernel<KC, RES, KN, true, FUSED>
              : p.sim == SPD_SIM_COS ? kmeans_kernel<KC, RES, KN, true> : kmeans_kernel<KC, RES, KN, false>;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(KC, p.n_tiles);
  cfg.blockDim = dim3(kmeans_threads<KN>());
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = KC;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kern, p, w, out);
}

const void* stream_kernel(int KC, int CG, bool cos) {
#define SPD_STREAM(kc)                                                                                  \
  if (KC == kc)                                                                                         \
    return CG == 1 ? (cos ? (const void*)kmeans_stream_kernel<kc, 1, true>                              \
                          : (const void*)kmeans_stream_kernel<kc, 1, false>)                            \
                   : (cos ? (const void*)kmeans_stream_kernel<kc, 2, true>                              \
                          : (const void*)kmeans_stream_kernel<kc, 2, false>);
  SPD_STREAM(1)
  SPD_STREAM(2)
  SPD_STREAM(4)
  SPD_STREAM(8)
#undef SPD_STREAM
  return nullptr;
}

// Kernel attributes (once per process) and whether 16-CTA clusters of the resident kernel fit.
int kmeans_setup() {
  static std::once_flag once;
  static cudaError_t err = cudaSuccess;
  std::call_once(once, [] {
    auto streamed = [](auto kern) {
      return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * 24576 * 4);
    };
    auto resident = [](auto kern) {
      cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
      if (e == cudaSuccess)
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kResSmem));
      return e;
    };
    err = streamed(kmeans_kernel<8, false, 4, true>);
    if (err == cudaSuccess) err = streamed(kmeans_kernel<8, false, SPD_MAX_CLUSTERS, true>);
    if (err == cudaSuccess) err = resident(kmeans_kernel<16, true, 4, true>);
    if (err == cudaSuccess) err = resident(kmeans_kernel<16, true, SPD_MAX_CLUSTERS, true>);
    if (err == cudaSuccess) err = streamed(kmeans_kernel<8, false, 4, false>);
    if (err == cudaSuccess) err = streamed(kmeans_kernel<8, false, SPD_MAX_CLUSTERS, false>);
    if (err == cudaSuccess) err = resident(kmeans_kernel<16, true, 4, false>);
    if (err == cudaSuccess) err = resident(kmeans_kernel<16, true, SPD_MAX_CLUSTERS, false>);
    if (err == cudaSuccess) err = resident(kmeans_kernel<16, true, 4, true, true>);
    if (err == cudaSuccess) err = resident(kmeans_kernel<16, true, SPD_MAX_CLUSTERS, true, true>);
    auto wide = [](auto kern) {
      return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kResSmem));
    };
    if (err == cudaSuccess) err = wide(kmeans_grid_kernel<4, true>);
    if (err == cudaSuccess) err = wide(kmeans_grid_kernel<4, false>);
    if (err == cudaSuccess) err = wide(kmeans_grid_kernel<SPD_MAX_CLUSTERS, true>);
    if (err == cudaSuccess) err = wide(kmeans_grid_kernel<SPD_MAX_CLUSTERS, false>);
    for (int i = 0; i < 16 && err == cudaSuccess; ++i)
      err = cudaFuncSetAttribute(stream_kernel(1 << (i & 3), i & 4 ? 2 : 1, i & 8),
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, int(kStreamSmem));
    g_res_clusters = 0;
    if (err == cudaSuccess) {
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(16);
      cfg.blockDim = dim3(512);
      cfg.dynamicSmemBytes = kResSmem;
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = 16;
      attr[0].val.clusterDim.y = 1;
      attr[0].val.clusterDim.z = 1;
      cfg.attrs = attr;
      cfg.numAttrs = 1;
      for (int kc = 2; kc <= 8 && err == cudaSuccess; kc *= 2) {
        cudaLaunchConfig_t sc = cfg;
        cudaLaunchAttribute sa[1];
        sc.gridDim = dim3(kc);
        sc.blockDim = dim3(kStreamThreads);
        sc.dynamicSmemBytes = kStreamSmem;
        sa[0].id = cudaLaunchAttributeClusterDimension;
        sa[0].val.clusterDim.x = kc;
        sa[0].val.clusterDim.y = 1;
        sa[0].val.clusterDim.z = 1;
        sc.attrs = sa;
        if (cudaOccupancyMaxActiveClusters(&g_stream_clusters[kc], stream_kernel(kc, 1, true), &sc) != cudaSuccess) {
          cudaGetLastError();
          g_stream_clusters[kc] = 0;
        }
      }
      int n = 0;
      if (cudaOccupancyMaxActiveClusters(&n, kmeans_kernel<16, true, SPD_MAX_CLUSTERS, true>, &cfg) !=
          cudaSuccess) {
        cudaGetLastError();
        n = 0;
      }
      g_res_clusters = n;
      g_grid_fits = true;
      for (const void* kern : {(const void*)kmeans_grid_kernel<4, true>, (const void*)kmeans_grid_kernel<4, false>,
                               (const void*)kmeans_grid_kernel<SPD_MAX_CLUSTERS, true>,
                               (const void*)kmeans_grid_kernel<SPD_MAX_CLUSTERS, false>}) {
        int blocks = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, kern, kGridThreads, kResSmem) != cudaSuccess)
          cudaGetLastError();
        if (blocks < 1) g_grid_fits = false;
      }
    }
  });
  if (err != cudaSuccess) return fail(SPD_ECUDA, "K-means attributes: %s", cudaGetErrorString(err));
  return SPD_OK;
}

// Which kernels spd_prune launches for p (after kmeans_setup).
struct PrunePlan {
  bool anchor_sim, res, fused;
  int grid;        // CTAs a tile of the whole-GPU K-means, 0: clusters
  bool grid_res;   // its rows fit in shared memory
  size_t grid_smem;
  int stream;      // CTAs a tile of the one-sweep K-means, 0: none
  int stream_slots;
  int launches;
};
// whole_gpu: false where a cooperative launch over every SM is not to be had.
PrunePlan prune_plan(const PruneDims& p, bool whole_gpu = g_grid_fits) {
  PrunePlan q;
  q.anchor_sim = p.n_anc > 0 && p.m > 0 && p.wa != 0.0f;
  // K-means: the rows resident in shared memory over 16 CTAs per tile where they fit and all tiles
  // run in one wave of such clusters (latency); else the whole GPU or the one-sweep form below; else
  // (K other than 4, or rows too wide for the one-sweep ring) re-read from L2 each pass by 8 CTAs
  q.res = p.m > 0 && res_bytes(p) <= kResSmem && g_res_clusters > 0 && p.n_tiles <= g_res_clusters;
  // resident rows and the cosine kind: scores, selection and compaction in the same kernel (CTA 0's
  // row buffer holds the m sort keys and the n kept flags by then)
  const size_t row_bytes = size_t((p.m + 15) / 16) * p.d * sizeof(float);
  q.fused = q.res && p.sim == SPD_SIM_COS && (p.m + 15) / 16 <= 512 &&
            row_bytes >= size_t(8) * (p.m + 1) + p.n;
  // Tiles whose rows do not fit the 16 CTAs of a cluster (or more tiles than such clusters), few enough
  // for 15 SMs each: the whole GPU. One image of 700 / 1024 / 2739 / 4096 x 1280: 199 / 279 / 671 / 976 ->
  // 104 / 135 / 204 / 330 us a call; 9 / 10 tiles of 576 x 1024: 170 / 176 -> 149 / 160 us, but 12 of
  // them 183 -> 187 us.
  q.grid = 0;
  if (!q.res && whole_gpu && grid_tile(p)) {
    const int G = std::min(num_sms() / p.n_tiles, grid_ctas(p));
    const size_t nl = (p.m + G - 1) / std::max(G, 1);
    if (G >= 15 && nl <= size_t(kGridMaxRows)) {
      q.grid = G;
      q.grid_smem = size_t(p.K) * p.d * sizeof(float);
      q.grid_res = q.grid_smem + nl * p.d * sizeof(float) <= kResSmem;
      if (q.grid_res) q.grid_smem += nl * p.d * sizeof(float);
    }
  }
  // Many tiles: one sweep an iteration, over as many CTAs a tile as the SMs hold at one each
  q.stream = 0;
  if (!q.res && !q.grid && p.K == 4 && p.d >= 64 && p.d <= 8 * kStreamThreads && p.m > 0) {
    int KC = 8;
    while (KC > 1 && p.n_tiles > g_stream_clusters[KC]) KC /= 2;
    q.stream_slots = std::min(3, stream_slots(p.d, (p.m + KC - 1) / KC, kStreamSmem));
    if (q.stream_slots >= 2) q.stream = KC;
  }
  q.launches = 2 + int(q.anchor_sim) + 1 + (q.fused ? 0 : int(p.m > 0) + 1);
  return q;
}

cudaError_t launch_stream(const PruneDims& p, const PruneWs& w, const PrunePlan& q, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(q.stream, p.n_tiles);
  cfg.blockDim = dim3(kStreamThreads);
  cfg.dynamicSmemBytes = kStreamSmem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = q.stream;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  using Fn = void (*)(PruneDims, PruneWs, int);
  auto kern = reinterpret_cast<Fn>(const_cast<void*>(stream_kernel(q.stream, stream_groups(p.d),
                                                                   p.sim == SPD_SIM_COS)));
  return cudaLaunchKernelEx(&cfg, kern, p, w, q.stream_slots);
}

}  // namespace
}  // namespace spd

using namespace spd;

extern "C" int spd_selftest_tile_barrier(void* ws, int barriers, long long budget_cycles, void* stream) {
  if (!ws || barriers < 1) return fail(SPD_EINVAL, "null workspace or no barriers");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  SPD_CUDA_TRY(cudaMemsetAsync(static_cast<int*>(ws) + 1, 0, sizeof(int), st));
  tile_barrier_probe_kernel<<<16, 32, 0, st>>>(static_cast<int*>(ws), barriers, budget_cycles);
  SPD_CUDA_TRY(cudaGetLastError());
  return SPD_OK;
}

extern "C" int spd_prune_launches(const spd_prune_cfg* cfg) {
  PruneDims p;
  if (int rc = validate(cfg, &p)) return rc;
  if (int rc = kmeans_setup()) return rc;
  return prune_plan(p).launches;
}

extern "C" size_t spd_prune_workspace_size(const spd_prune_cfg* cfg) {
  PruneDims p;
  if (validate(cfg, &p)) return 0;
  Carve cv(nullptr, ~size_t(0));
  carve(p, cv);
  return cv.used;
}

extern "C" int spd_prune(const spd_prune_cfg* cfg, const float* const* feats, const float* attn,
                         int32_t* keep_idx, uint8_t* kind, int8_t* cluster, float* scores, void* ws,
                         size_t ws_bytes, void* stream_) {
  PruneDims p;
  if (int rc = validate(cfg, &p)) return rc;
  if (!feats || !attn || !keep_idx || !ws) return fail(SPD_EINVAL, "null buffer");
  for (int l = 0; l < p.L; ++l) {
    if (!feats[l] || (reinterpret_cast<uintptr_t>(feats[l]) & 15))
      return fail(SPD_EINVAL, "feature pointer %d null or not 16-byte aligned", l);
    p.feat[l] = feats[l];
  }
  Carve cv(ws, ws_bytes);
  PruneWs w = carve(p, cv);
  if (!cv.fits()) return fail(SPD_ENOSPC, "prune workspace too small (%zu < %zu)", ws_bytes, cv.used);
  cudaStream_t st = static_cast<cudaStream_t>(stream_);
  const int T = p.n_tiles;
  const int slot = trace_begin(st);
  SPD_CUDA_TRY(launch_pdl_carveout(kPruneCarveout, p.sim == SPD_SIM_COS ? rowstats_kernel<SPD_SIM_COS>
                          : p.sim == SPD_SIM_MSE ? rowstats_kernel<SPD_SIM_MSE> : rowstats_kernel<SPD_SIM_KL>,
                          dim3((p.n + 7) / 8, T), dim3(256), 0, st, p, attn, w));
  SPD_CUDA_TRY(launch_pdl_carveout(kPruneCarveout, anchor_kernel, dim3(rank_ctas(p.n), T), dim3(kRankThreads), 0, st,
                                   p, w));
  if (int rc = kmeans_setup()) return rc;
  PrunePlan plan = prune_plan(p);
  if (plan.anchor_sim) {
    const int aw = (p.n_anc + 47) / 48 * 48 < (p.n_anc + 63) / 64 * 64 ? 48 : 64;
    const int ay = (p.n_anc + aw - 1) / aw;
    const size_t ctas = size_t((p.m + 127) / 128) * ay * T * 8;  // at R = 128, AS = 8
    const int as = ctas <= 3 * size_t(num_sms()) ? 8 : 4, rows = ctas < size_t(num_sms()) ? 64 : 128;
    const dim3 g((p.m + rows - 1) / rows, ay, T);
    auto pick = [&](auto sim) {
      constexpr int S = decltype(sim)::value;
      return rows == 64 ? (aw == 48 ? anchor_sim_kernel<S, 8, 48, 64> : anchor_sim_kernel<S, 8, 64, 64>)
             : as == 8  ? (aw == 48 ? anchor_sim_kernel<S, 8, 48, 128> : anchor_sim_kernel<S, 8, 64, 128>)
                        : (aw == 48 ? anchor_sim_kernel<S, 4, 48, 128> : anchor_sim_kernel<S, 4, 64, 128>);
    };
    auto kern = p.sim == SPD_SIM_COS   ? pick(std::integral_constant<int, SPD_SIM_COS>())
                : p.sim == SPD_SIM_MSE ? pick(std::integral_constant<int, SPD_SIM_MSE>())
                                       : pick(std::integral_constant<int, SPD_SIM_KL>());
    SPD_CUDA_TRY(launch_pdl_carveout(kPruneCarveout, kern, dim3(g.x * as, g.y, T), dim3(256), 0, st, p, w));
  }
  const size_t cent_bytes = size_t(2) * p.K * p.d * sizeof(float);
  const PruneOut out{keep_idx, kind, cluster, scores};
  if (plan.grid) {
    auto kern = p.K == 4 ? (p.sim == SPD_SIM_COS ? kmeans_grid_kernel<4, true> : kmeans_grid_kernel<4, false>)
                : p.sim == SPD_SIM_COS ? kmeans_grid_kernel<SPD_MAX_CLUSTERS, true>
                                       : kmeans_grid_kernel<SPD_MAX_CLUSTERS, false>;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(plan.grid * T);
    cfg.blockDim = dim3(kGridThreads);
    cfg.dynamicSmemBytes = plan.grid_smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];  // every CTA resident: they wait on one another
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, p, w, plan.grid, int(plan.grid_res));
    if (e == cudaErrorCooperativeLaunchTooLarge) {  // the stream's context has fewer SMs than the device
      cudaGetLastError();
      plan = prune_plan(p, false);
    } else {
      SPD_CUDA_TRY(e);
    }
  }
  if (plan.grid) {
    // launched above
  } else if (plan.fused && p.K == 4)
    SPD_CUDA_TRY((launch_kmeans<16, true, 4, true>(p, w, out, res_bytes(p), st)));
  else if (plan.fused)
    SPD_CUDA_TRY((launch_kmeans<16, true, SPD_MAX_CLUSTERS, true>(p, w, out, res_bytes(p), st)));
  else if (plan.res && p.K == 4)
    SPD_CUDA_TRY((launch_kmeans<16, true, 4>(p, w, out, res_bytes(p), st)));
  else if (plan.res)
    SPD_CUDA_TRY((launch_kmeans<16, true, SPD_MAX_CLUSTERS>(p, w, out, res_bytes(p), st)));
  else if (plan.stream)
    SPD_CUDA_TRY(launch_stream(p, w, plan, st));
  else if (p.K == 4)
    SPD_CUDA_TRY((launch_kmeans<8, false, 4>(p, w, out, cent_bytes, st)));
  else
    SPD_CUDA_TRY((launch_kmeans<8, false, SPD_MAX_CLUSTERS>(p, w, out, cent_bytes, st)));
  if (!plan.fused) {
    if (p.m > 0) {
      auto score = p.sim == SPD_SIM_COS ? score_kernel<SPD_SIM_COS>
                   : p.sim == SPD_SIM_MSE ? score_kernel<SPD_SIM_MSE> : score_kernel<SPD_SIM_KL>;
      SPD_CUDA_TRY(launch_pdl_carveout(kPruneCarveout, score, dim3((p.m + 7) / 8, T), dim3(256), 0, st, p, w));
    }
    SPD_CUDA_TRY(launch_pdl_carveout(kPruneCarveout, select_kernel, dim3(rank_ctas(p.m), T), dim3(kRankThreads), 0, st,
                                     p, w, keep_idx, kind, cluster, scores));
  }
  // algorithmic work per tile: every tapped layer's features and the attention read once, the
  // kept indices written; anchor similarities (n - N_anc) N_anc d multiply-adds
  trace_end(slot, st, TR_PRUNE, 2.0 * T * double(p.m) * p.n_anc * p.d,
            T * (4.0 * p.L * double(p.n_tok) * p.d + 4.0 * p.H * p.n_att + 4.0 * p.keep + 6.0 * p.n));
  return SPD_OK;
}

namespace {
int received_splits(int n_maps, int n_q, int n_k) {
  const int blocks = (n_k / 4 + 255) / 256;
  // About four CTAs an SM (32 KB of loads in flight each): with two, 2.1 a SM at 16 maps of 3840 x 3840 left
  // half of the SMs at two thirds of the others' share, 183 us against 138 (6.8 TB/s); eight were slower at
  // 32 maps of 4096 x 4096 (350 us, 303 at four).
  int sp = (4 * num_sms() + blocks * n_maps - 1) / (blocks * n_maps);
  sp = std::max(1, std::min(sp, (n_q + 63) / 64));                    // at least 64 rows each
  return sp;
}
}  // namespace

extern "C" size_t spd_received_attention_workspace_size(int n_maps, int n_q, int n_k) {
  if (n_maps < 1 || n_q < 1 || n_k < 4) return 0;
  Carve cv(nullptr, ~size_t(0));
  cv.take<float>(size_t(received_splits(n_maps, n_q, n_k)) * n_maps * n_k);
  return cv.used;
}

extern "C" int spd_received_attention(const float* maps, int n_maps, int n_q, int n_k,
                                      const int32_t* group_start, const int32_t* group_members,
                                      int n_out, float* out, void* ws, size_t ws_bytes,
                                      void* stream_) {
  if (!maps || !out || !ws || n_maps < 1 || n_q < 1 || n_k < 4 || n_k % 4 ||
      (reinterpret_cast<uintptr_t>(maps) & 15))
    return fail(SPD_EINVAL, "bad received-attention arguments (n_k a multiple of 4, maps 16-byte aligned)");
  if ((group_start == nullptr) != (group_members == nullptr))
    return fail(SPD_EINVAL, "group_start and group_members go together");
  if (!group_start && n_out != n_k) return fail(SPD_EINVAL, "without groups n_out must equal n_k");
  if (n_out < 1) return fail(SPD_EINVAL, "n_out >= 1 required");
  const int sp = received_splits(n_maps, n_q, n_k);
  Carve cv(ws, ws_bytes);
  float* partial = cv.take<float>(size_t(sp) * n_maps * n_k);
  if (!cv.fits()) return fail(SPD_ENOSPC, "received-attention workspace too small");
  cudaStream_t st = static_cast<cudaStream_t>(stream_);
  const int rows = (n_q + sp - 1) / sp;
  const int slot = trace_begin(st);
  SPD_CUDA_TRY(launch_pdl(received_colsum_kernel, dim3((n_k / 4 + 255) / 256, n_maps, sp), dim3(256),
                          0, st, maps, n_q, n_k, rows, partial));
  SPD_CUDA_TRY(launch_pdl(received_finish_kernel, dim3((n_out + 255) / 256, n_maps), dim3(256), 0, st,
                          static_cast<const float*>(partial), n_maps, n_k, sp, float(1.0 / n_q),
                          group_start, group_members, n_out, out, cv.status()));
  // algorithmic work: every map entry read once, the result written once
  trace_end(slot, st, TR_PRUNE, double(n_maps) * n_q * n_k,
            4.0 * double(n_maps) * n_q * n_k + 4.0 * double(n_maps) * n_out);
  return SPD_OK;
}

extern "C" int spd_gather_rows_bf16(const float* src, int n_tiles, int n_tok, int d, int row_offset,
                                    const int32_t* idx, int keep, uint16_t* dst, void* ws,
                                    void* stream_) {
  if (!src || !idx || !dst || n_tiles < 1 || keep < 1 || d < 4 || d % 4 || row_offset < 0 ||
      row_offset >= n_tok)
    return fail(SPD_EINVAL, "bad gather arguments");
  SPD_CUDA_TRY(launch_pdl(gather_bf16_kernel, dim3(keep, n_tiles), dim3(128), 0,
                          static_cast<cudaStream_t>(stream_), src, n_tok, d, row_offset, idx, keep,
                          reinterpret_cast<__nv_bfloat16*>(dst), ws ? static_cast<int*>(ws) : nullptr));
  return SPD_OK;
}
