// Variable-length causal attention over packed sequences on the tcgen05 tensor cores, queries
// restricted to the attention-active tokens (VSkip-Attn, Sec. 3.2: a skipped token is not a
// query, but it stays a key and a value for every other token of its sequence).
//
// One CTA = up to 128 active queries of one sequence x one head (the MMA's M = 128 rows), two CTAs an SM:
//   warp 4     TMA producer: the Q tile once, then blocks of 64 keys of K and of V into two-stage rings
//              (128-byte swizzle, boxes of 64 head-dim columns)
//   warp 5     MMA issuer: S = Q K^T into TMEM (kind::f16, fp32), then O += P V with P read from TMEM and V
//              read in place as an MN-major operand (the layout its TMA box has)
//   warps 0-3  softmax: thread r owns query row r (TMEM lane r); one pass over the block's 64 scores in
//              registers, online softmax in fp32 with exp2, P rounded to bf16 over S's own TMEM columns, the
//              row sum over the unrounded weights; O is rescaled in TMEM when a row's maximum grew; at the
//              end O / l goes to HBM in bf16
// S alternates between two TMEM buffers, so S of block j + 1 is computed while the softmax of block j
// runs. A query at position p sees keys 0..p of its own sequence; tiles run from the last to the first (in
// causal order the longest first), all heads of a tile side by side. Every wait is bounded (status
// SPD_ETIMEOUT, no hang).
//
// What bounds it: a 64-key block is 640 cycles of tensor work (the S products are limited by the operand reads
// from shared memory), 512 of exponentials and about 300 instructions a softmax thread; the CTAs of an SM fill
// each other's waits. With one CTA of 128-key blocks an SM (P through shared memory, two passes over S, a
// rescale at every new maximum) the tensor pipe idled through each softmax: four requests of 1021-3302
// tokens, 28 heads of 128, 492 us; so 250 us (0.45 of the burst bf16 rate, counting the causal half only).
// Rescaling only where a maximum doubled and adding up the rounded weights took 244 us, at the price of weights
// up to 2 and of sums of 16-bit values; relative error against 64 bits 2.029e-3 (2.037e-3 with 128-key blocks).
#include <cuda_bf16.h>
#include <math.h>
#include <stdint.h>

#include <cooperative_groups.h>

#include "internal.h"
#include "ptx.cuh"
#include "trace.h"

namespace spd {
namespace {

namespace cg = cooperative_groups;

constexpr int kTK = 64;                // keys per block (S columns, K of the PV product)
constexpr uint32_t kQBox = 128 * 128;  // one TMA box of Q: 128 rows x 64 bf16
constexpr uint32_t kKBox = kTK * 128;  // ... of K and V: 64 rows
constexpr int kThreads = 192;
constexpr uint32_t kTmemCols = 256;    // S: two buffers [0, 64) and [64, 128); O: [128, 128 + HD)

template <int HD>
struct AttnSmem {
  static constexpr int kChunks = HD / 64;                       // 64-column boxes per row
  static constexpr uint32_t q = 0;                              // Q tile
  static constexpr uint32_t k = q + kChunks * kQBox;            // K stages
  static constexpr uint32_t v = k + 2 * kChunks * kKBox;        // V stages
  static constexpr uint32_t bars = v + 2 * kChunks * kKBox;
  static constexpr uint32_t bytes = bars + 128 + 1024;          // + alignment slack
};

__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}

template <int HD>
__global__ void __launch_bounds__(kThreads, 2)
    attn_tc_kernel(const __grid_constant__ CUtensorMap map_q,
                   const __grid_constant__ CUtensorMap map_kv, __nv_bfloat16* __restrict__ o,
                   int ldo, const int4* tiles, int n_tiles, const int32_t* q_pos, int n_heads, int n_kv_heads,
                   int v_off, float scale_log2, int* status, long long budget,
                   unsigned long long* stamp) {
  using L = AttnSmem<HD>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~uintptr_t(1023));
  uint64_t* q_full = reinterpret_cast<uint64_t*>(smem + L::bars);
  uint64_t* k_full = q_full + 1;   // [2] K block landed
  uint64_t* k_empty = q_full + 3;  // [2] its S product has completed
  uint64_t* v_full = q_full + 5;   // [2] V block landed
  uint64_t* v_empty = q_full + 7;  // [2] its PV product has completed
  uint64_t* s_full = q_full + 9;   // [2] S of block j is in TMEM buffer j % 2
  uint64_t* p_full = q_full + 11;  // [2] P of block j written (S read) and O rescaled; two, since a softmax
                                   // warp may finish block j + 1 before another has finished block j
  uint64_t* o_done = q_full + 13;  // PV product of the current block completed
  uint64_t* drain = q_full + 14;   // every MMA completed: O is final
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(q_full + 15);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int h = blockIdx.x % n_heads, tile = n_tiles - 1 - int(blockIdx.x) / n_heads;
  const int hk = h / (n_heads / n_kv_heads);
  if (threadIdx.x == 0) {
    mbar_init(q_full, 1);
    for (int s = 0; s < 2; ++s) {
      mbar_init(&k_full[s], 1);
      mbar_init(&k_empty[s], 1);
      mbar_init(&v_full[s], 1);
      mbar_init(&v_empty[s], 1);
      mbar_init(&s_full[s], 1);
      mbar_init(&p_full[s], 4);  // one arrival per softmax warp
    }
    mbar_init(o_done, 1);
    mbar_init(drain, 1);
    *abort_flag = 0;
    fence_mbar_init();
    prefetch_tmap(&map_q);
    prefetch_tmap(&map_kv);
  }
  if (warp == 4) {
    tmem_alloc(tmem_slot, kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const uint32_t t_o = tmem + 2 * kTK;  // S buffer b at tmem + 64 b

  // Nothing written by an earlier kernel of the stream is read before the grid dependency wait:
  // under programmatic overlap this kernel's prologue may run while several earlier kernels are
  // still resident, so the tile list and the positions (copied or built by a kernel) are read
  // after it, with coherent loads. Q, K and V come from the previous kernels too.
  pdl_launch_dependents();
  pdl_wait();
  if (threadIdx.x == 0) stamp_start(stamp);
  const int4 tl = tiles[tile];
  const int q0 = tl.x, nq = tl.y, kv0 = tl.z, len = tl.w;
  if (nq == 0) {  // padding of a list made on the device: nothing to do
    if (warp == 4) tmem_dealloc(tmem, kTmemCols);
    if (threadIdx.x == 0) stamp_end(stamp);
    return;
  }
  const int p_last = q_pos[q0 + nq - 1];  // positions ascend within a tile
  const int nkb = max(1, min((p_last + kTK) / kTK, (len + kTK - 1) / kTK));
  const int my_pos = threadIdx.x < 128 ? q_pos[q0 + min(int(threadIdx.x), nq - 1)] : 0;

  int issued_k = 0, issued_v = 0;  // blocks whose loads the producer issued
  if (warp == 4) {
    if (lane == 0) {
      // ---- TMA producer ----
      const uint64_t pol_q = policy_evict_first(), pol_kv = policy_evict_last();
      mbar_arrive_expect_tx(q_full, L::kChunks * kQBox);
      for (int c = 0; c < L::kChunks; ++c)
        tma_load_2d(smem + L::q + c * kQBox, &map_q, q_full, h * HD + c * 64, q0, pol_q);
      auto load = [&](int j, uint64_t* full, uint64_t* empty, uint32_t at, int x0) -> bool {
        const int s = j & 1;
        if (j >= 2 && !mbar_wait(&empty[s], ((j >> 1) - 1) & 1, abort_flag, budget)) {
          *abort_flag = 1;
          set_status(status, SPD_ETIMEOUT);
          return false;
        }
        mbar_arrive_expect_tx(&full[s], L::kChunks * kKBox);
        for (int c = 0; c < L::kChunks; ++c)
          tma_load_2d(smem + at + (s * L::kChunks + c) * kKBox, &map_kv, &full[s], x0 + hk * HD + c * 64,
                      kv0 + j * kTK, pol_kv);
        return true;
      };
      for (int j = 0; j < nkb; ++j) {
        if (!load(j, k_full, k_empty, L::k, 0)) break;
        issued_k = j + 1;
        if (!load(j, v_full, v_empty, L::v, v_off)) break;
        issued_v = j + 1;
      }
    }
  } else if (warp == 5) {
    if (lane == 0) {
      // ---- MMA issuer ----
      const uint32_t id_s = idesc_bf16_f32(128, kTK);
      const uint32_t id_o = idesc_bf16_f32(128, HD) | (1u << 16);  // V is MN-major
      const uint32_t sq = smem_u32(smem + L::q);
      bool ok = mbar_wait(q_full, 0, abort_flag, budget);
      auto issue_s = [&](int j) -> bool {
        const int s = j & 1;
        if (!mbar_wait(&k_full[s], (j >> 1) & 1, abort_flag, budget)) return false;
        // S buffer s holds P of block j - 2 until its PV product has completed
        if (j > 1 && !mbar_wait(o_done, j & 1, abort_flag, budget)) return false;
        tc_fence_after();
        const uint32_t sk = smem_u32(smem + L::k + s * L::kChunks * kKBox);
#pragma unroll
        for (int kk = 0; kk < HD / 16; ++kk)
          mma_bf16(tmem + kTK * s, sdesc_k128(sq + (kk >> 2) * kQBox + (kk & 3) * 32),
                   sdesc_k128(sk + (kk >> 2) * kKBox + (kk & 3) * 32), id_s, kk > 0 ? 1u : 0u);
        mma_commit(&s_full[s]);
        mma_commit(&k_empty[s]);
        return true;
      };
      if (ok) ok = issue_s(0);
      for (int j = 0; j < nkb && ok; ++j) {
        const int s = j & 1;
        if (j + 1 < nkb && !(ok = issue_s(j + 1))) break;
        if (!(ok = mbar_wait(&v_full[s], (j >> 1) & 1, abort_flag, budget))) break;
        if (!(ok = mbar_wait(&p_full[s], (j >> 1) & 1, abort_flag, budget))) break;
        tc_fence_after();
        const uint32_t sv = smem_u32(smem + L::v + s * L::kChunks * kKBox);
#pragma unroll
        for (int kk = 0; kk < kTK / 16; ++kk)
          mma_bf16_ts(t_o, tmem + kTK * s + 8 * kk, sdesc_mn128(sv + kk * 2048, kKBox), id_o,
                      (j > 0 || kk > 0) ? 1u : 0u);
        mma_commit(o_done);
        mma_commit(&v_empty[s]);
      }
      if (!ok) {
        *abort_flag = 1;
        set_status(status, SPD_ETIMEOUT);
      }
      mma_commit(drain);  // arrives once every MMA issued above has completed
      volatile int no_abort = 0;
      if (!mbar_wait(drain, 0, &no_abort, budget)) set_status(status, SPD_ETIMEOUT);
    }
  } else {
    // ---- softmax and epilogue: warp w reads TMEM lanes [32 w, 32 w + 32) ----
    const int r = warp * 32 + lane;  // query row of the tile
    const uint32_t lanes = static_cast<uint32_t>(warp * 32) << 16;
    float m_run = -INFINITY, l_run = 0.0f;  // the row's maximum so far (raw scores) and sum of weights
    const int pos_min = __shfl_sync(0xffffffffu, my_pos, 0);  // the warp's first row sees the fewest keys
    bool ok = true;
    for (int j = 0; j < nkb; ++j) {
      const uint32_t t_s = tmem + kTK * (j & 1) + lanes;
      if (!(ok = __all_sync(0xffffffffu, mbar_wait(&s_full[j & 1], (j >> 1) & 1, abort_flag, budget))))
        break;
      tc_fence_after();
      float v[kTK];
      tmem_ld64(t_s, v);
      const int kb = j * kTK;
      if (pos_min < kb + kTK - 1) {  // some row of the warp does not see the whole block (warp-uniform)
#pragma unroll
        for (int i = 0; i < kTK; ++i)
          if (kb + i > my_pos) v[i] = -INFINITY;
      }
      float m4[4] = {v[0], v[1], v[2], v[3]};
#pragma unroll
      for (int i = 4; i < kTK; ++i) m4[i & 3] = fmaxf(m4[i & 3], v[i]);
      const float mx = fmaxf(fmaxf(m4[0], m4[1]), fmaxf(m4[2], m4[3]));
      if (j == 0) {
        m_run = mx;  // finite: block 0 holds key 0 <= every position
      } else if (__any_sync(0xffffffffu, mx > m_run)) {
        // the previous PV product has completed (the one before it had when these scores came): O can be
        // rescaled
        if (!(ok = __all_sync(0xffffffffu, mbar_wait(o_done, (j - 1) & 1, abort_flag, budget))))
          break;
        tc_fence_after();
        const float m_new = fmaxf(m_run, mx);
        const float corr = ex2((m_run - m_new) * scale_log2);
        m_run = m_new;
        l_run *= corr;
#pragma unroll 1
        for (int c = 0; c < HD / 32; ++c) {
          float ov[32];
          tmem_ld32(t_o + lanes + c * 32, ov);
#pragma unroll
          for (int i = 0; i < 32; ++i) ov[i] *= corr;
          tmem_st32(t_o + lanes + c * 32, ov);
        }
      }
      const float off = m_run * scale_log2;
      float r4[4] = {0.0f, 0.0f, 0.0f, 0.0f};
      uint32_t pk[kTK / 2];
#pragma unroll
      for (int i = 0; i < kTK; i += 2) {
        const float p0 = ex2(fmaf(v[i], scale_log2, -off)), p1 = ex2(fmaf(v[i + 1], scale_log2, -off));
        r4[i & 2] += p0;
        r4[(i & 2) + 1] += p1;
        pk[i >> 1] = pack_bf16(p0, p1);
      }
      l_run += (r4[0] + r4[1]) + (r4[2] + r4[3]);
      float pf[32];
#pragma unroll
      for (int i = 0; i < 32; ++i) pf[i] = __uint_as_float(pk[i]);
      tmem_st32(t_s, pf);  // over the scores: keys 2 i and 2 i + 1 in column i
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&p_full[j & 1]);
    }
    // (not o_done: here its phase may be any of the last two, which a parity cannot tell apart)
    if (ok) ok = __all_sync(0xffffffffu, mbar_wait(drain, 0, abort_flag, budget));
    if (!ok) {
      *abort_flag = 1;
      set_status(status, SPD_ETIMEOUT);
    } else {
      tc_fence_after();
      const float inv = 1.0f / l_run;
      __nv_bfloat16* orow = o + size_t(q0 + r) * ldo + h * HD;
#pragma unroll 1
      for (int c = 0; c < HD / 32; ++c) {
        float v[32];
        tmem_ld32(t_o + lanes + c * 32, v);
        if (r < nq) {
#pragma unroll
          for (int u = 0; u < 4; ++u)
            reinterpret_cast<uint4*>(orow + c * 32)[u] =
                make_uint4(pack_bf16(v[8 * u] * inv, v[8 * u + 1] * inv),
                           pack_bf16(v[8 * u + 2] * inv, v[8 * u + 3] * inv),
                           pack_bf16(v[8 * u + 4] * inv, v[8 * u + 5] * inv),
                           pack_bf16(v[8 * u + 6] * inv, v[8 * u + 7] * inv));
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 128 && *abort_flag) {
    // loads issued but never consumed land before the CTA exits (without an abort the last products
    // consumed every issued block)
    volatile int no_abort = 0;
    mbar_wait(q_full, 0, &no_abort, budget);
    for (int j = max(0, issued_k - 2); j < issued_k; ++j) mbar_wait(&k_full[j & 1], (j >> 1) & 1, &no_abort, budget);
    for (int j = max(0, issued_v - 2); j < issued_v; ++j) mbar_wait(&v_full[j & 1], (j >> 1) & 1, &no_abort, budget);
  }
  __syncwarp();
  tc_fence_after();
  if (warp == 4) tmem_dealloc(tmem, kTmemCols);
  if (threadIdx.x == 0) stamp_end(stamp);
}

template <int HD>
int launch(const CUtensorMap& mq, const CUtensorMap& mkv, void* o, int ldo, const int4* tiles,
           int n_tiles, const int32_t* q_pos, int n_heads, int n_kv_heads, int v_off, int* status,
           cudaStream_t stream, unsigned long long* stamp) {
  using L = AttnSmem<HD>;
  static bool attr = false;
  if (!attr) {
    SPD_CUDA_TRY(cudaFuncSetAttribute(attn_tc_kernel<HD>,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize, int(L::bytes)));
    attr = true;
  }
  const float scale_log2 = 1.4426950408889634f / sqrtf(float(HD));
  SPD_CUDA_TRY(launch_pdl(attn_tc_kernel<HD>, dim3(n_tiles * n_heads), dim3(kThreads), L::bytes,
                          stream, mq, mkv, static_cast<__nv_bfloat16*>(o), ldo, tiles, n_tiles, q_pos,
                          n_heads, n_kv_heads, v_off, scale_log2, status, kWaitBudget, stamp));
  return SPD_OK;
}

// ---- one query per sequence (a decode step) ---------------------------------------------------
// One CTA = a contiguous share of one sequence's keys x up to eight query heads of one K/V head, so K
// and V leave L2 once for all the heads that read them; a cluster of S CTAs (attention_decode_run)
// covers the sequence. The step is bound by the K/V stream (a token and layer: 4 n_kv_heads HD
// bytes), so all that matters is many wide loads in flight and few instructions a key: each of the
// eight warps takes groups of 16 keys, 16 bytes a lane and load, and multiplies them with the legacy
// m16n8k16 tensor instruction straight from registers (at most 8 of a tile's 128 rows would be
// queries on the tcgen05 path, which would also have to stage K and V in shared memory).
// Eight warps of 224 registers, one CTA an SM: four CTAs of four warps were slower (a whole step of one sequence
// 3167 against 3142 us), two CTAs of 128 registers spill and are no faster (64 sequences of 500 keys, 32 heads, four
// layers: 1069 us both), and without the second launch bound the compiler takes 207 registers and 1162 us.
// One layer's attention of 32 sequences (28 query heads on 4 K/V heads of 128, 1122 keys on average,
// 73 MB, serialised): 143 us with one warp a key and one CTA a query head, 35.5 us so and 29 with the
// longest sequences first; the step of four layers 1256 -> 829 us. One sequence of 257 keys, 32 heads: 10.4 -> 7.2 us.
//  * S = Q K^T: heads are the 16 rows of A (rows 8..15 stay zero), keys the 8 columns of B. The
//    order of the contraction index is free, so lane (r = lane / 4, c = lane % 4) feeds the two
//    MMAs of a 32-dim block from one 16-byte load of key r, dims 8 c .. 8 c + 7, of K and of Q alike. Each MMA
//    starts from zero and the sums are fp32 additions: a chain would lose its low bits.
//  * O += P V: P is split into three bf16 terms, which hold all 24 bits of it: the first, hi, in rows 0..7 of two
//    MMAs, half of it each, the others in rows 8..15 of the first and of the second. (hi has rows of its own
//    since the others may be zero or negative, which an infinite V must not meet.) V of key k, dims
//    8 r .. 8 r + 7 is one 16-byte load, byte-permuted into pairs of keys.
// Error of the bf16 outputs against 64 bits, 12 shapes of 257 to 2047 keys, four seeds each: the same to seven digits
// as with fp32 FMAs, and as many outputs at a border that round the other way (0.01 to 0.05 %; 0.05 to 0.2 %
// with two terms and chained sums, which held 17 bits of P). The third term and the sums from zero change a step of
// one sequence from 2842 to 2831 us, of 32 from 768 to 760, with 32 K/V heads of 10 / 16 / 64 sequences of 900 / 900 /
// 500 keys from 608 / 642 / 1028 to 577 / 648 / 1069.
// Online softmax a warp (running maximum m, sum l), O rescaled only when some maximum grew. The
// warps' states are merged in warp order, the CTAs' in rank order through distributed shared memory,
// each CTA finishing a share of the outputs.
constexpr int kDecWarps = 8;
constexpr int kDecHeads = 8;     // query heads a CTA
constexpr int kDecMaxSplit = 8;  // CTAs a cluster

// Eight bf16 of a K/V row; A16: the address is 16-byte aligned (else 4-byte).
template <bool A16>
__device__ __forceinline__ uint4 load8(const __nv_bfloat16* p) {
  if constexpr (A16) {
    return *reinterpret_cast<const uint4*>(p);
  } else {
    const uint32_t* w = reinterpret_cast<const uint32_t*>(p);
    return make_uint4(w[0], w[1], w[2], w[3]);
  }
}

template <int HD, bool A16>
__global__ void __launch_bounds__(kDecWarps * 32, 1)
    attn_decode_kernel(const __nv_bfloat16* q, const __nv_bfloat16* kv, int ldkv, int v_off,
                       __nv_bfloat16* __restrict__ o, int ldo, const int4* tiles, int n_heads,
                       int n_kv_heads, int chunks, float scale_log2, unsigned long long* stamp) {
  constexpr int KB = HD / 32, VB = HD / 64;  // 16-byte loads of a lane per key: K, V
  __shared__ float wm[kDecWarps][kDecHeads], wl[kDecWarps][kDecHeads];
  __shared__ float wo[kDecWarps][kDecHeads][HD];
  __shared__ float cm[kDecHeads], cl[kDecHeads], co[kDecHeads][HD];  // this CTA's merged state
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = int(cluster.block_rank()), S = int(cluster.num_blocks());
  pdl_launch_dependents();
  pdl_wait();
  if (threadIdx.x == 0) stamp_start(stamp);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, r = lane >> 2, c = lane & 3;
  // all heads of a sequence side by side, the sequences in the list's order
  const int groups = n_kv_heads * chunks, seq = blockIdx.x / groups, grp = blockIdx.x - seq * groups;
  const int G = n_heads / n_kv_heads, g = grp / chunks, hc = (grp - g * chunks) * kDecHeads;
  const int h0 = g * G + hc, ng = min(kDecHeads, G - hc);
  const int4 tl = tiles[seq];  // (query row, query count = 1, first key row, key count)
  const int j_lo = int((long long)rank * tl.w / S), j_hi = int((long long)(rank + 1) * tl.w / S);
  const __nv_bfloat16* kbase = kv + size_t(tl.z) * ldkv + g * HD;
  uint4 qf[KB];
#pragma unroll
  for (int i = 0; i < KB; ++i)
    qf[i] = r < ng ? *reinterpret_cast<const uint4*>(q + size_t(tl.x) * (n_heads * HD) + (h0 + r) * HD + 32 * i + 8 * c)
                   : make_uint4(0u, 0u, 0u, 0u);
  float m = -INFINITY, l = 0.0f;
  float acc[VB][8][4];  // rows r (hi) and r + 8 (the rest), dims 64 b + 16 c + j and 64 b + 16 c + 8 + j
#pragma unroll
  for (int b = 0; b < VB; ++b)
#pragma unroll
    for (int j = 0; j < 8; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[b][j][e] = 0.0f;
  for (int k0 = j_lo + 16 * warp; k0 < j_hi; k0 += 16 * kDecWarps) {
    // keys past the share load as zeros (their weight is zero, and 0 x 0 stays 0)
    uint4 kf[2][KB], vf[4][VB];
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      const int key = k0 + 8 * t + r;
#pragma unroll
      for (int i = 0; i < KB; ++i)
        kf[t][i] = key < j_hi ? load8<A16>(kbase + size_t(key) * ldkv + 32 * i + 8 * c) : make_uint4(0u, 0u, 0u, 0u);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int key = k0 + 8 * (u >> 1) + 2 * c + (u & 1);
#pragma unroll
      for (int b = 0; b < VB; ++b)
        vf[u][b] = key < j_hi ? load8<A16>(kbase + size_t(key) * ldkv + v_off + 64 * b + 8 * r)
                              : make_uint4(0u, 0u, 0u, 0u);
    }
    float s[2][2] = {{0.0f, 0.0f}, {0.0f, 0.0f}};
#pragma unroll
    for (int i = 0; i < KB; ++i)
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        float p0[4] = {0.0f, 0.0f, 0.0f, 0.0f}, p1[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        mma_16816(p0, qf[i].x, 0u, qf[i].y, 0u, kf[t][i].x, kf[t][i].y);
        mma_16816(p1, qf[i].z, 0u, qf[i].w, 0u, kf[t][i].z, kf[t][i].w);
        s[t][0] += p0[0] + p1[0];
        s[t][1] += p0[1] + p1[1];
      }
    // head r, keys k0 + 2 c + {0, 1} and k0 + 8 + 2 c + {0, 1}
    float x[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int key = k0 + 8 * (u >> 1) + 2 * c + (u & 1);
      x[u] = key < j_hi ? s[u >> 1][u & 1] * scale_log2 : -INFINITY;
    }
    float mx = fmaxf(fmaxf(x[0], x[1]), fmaxf(x[2], x[3]));
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
    const float mn = fmaxf(m, mx);  // finite: key k0 lies in the share
    if (__any_sync(0xffffffffu, mn != m)) {
      const float corr = exp2f(m - mn);
      l *= corr;
#pragma unroll
      for (int b = 0; b < VB; ++b)
#pragma unroll
        for (int j = 0; j < 8; ++j)
#pragma unroll
          for (int e = 0; e < 4; ++e) acc[b][j][e] *= corr;
      m = mn;
    }
    float hi[4], lo[4], rem[4];  // half of the first term; the others
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const float p = exp2f(x[u] - m), first = __bfloat162float(__float2bfloat16_rn(p));
      l += p;
      hi[u] = 0.5f * first;
      lo[u] = p - first;
      rem[u] = lo[u] - __bfloat162float(__float2bfloat16_rn(lo[u]));
    }
    const uint32_t a0 = pack_bf16(hi[0], hi[1]), a2 = pack_bf16(hi[2], hi[3]);
    const uint32_t a1 = pack_bf16(lo[0], lo[1]), a3 = pack_bf16(lo[2], lo[3]);
    const uint32_t c1 = pack_bf16(rem[0], rem[1]), c3 = pack_bf16(rem[2], rem[3]);
#pragma unroll
    for (int b = 0; b < VB; ++b) {
      const uint32_t w[4][4] = {{vf[0][b].x, vf[0][b].y, vf[0][b].z, vf[0][b].w},
                                {vf[1][b].x, vf[1][b].y, vf[1][b].z, vf[1][b].w},
                                {vf[2][b].x, vf[2][b].y, vf[2][b].z, vf[2][b].w},
                                {vf[3][b].x, vf[3][b].y, vf[3][b].z, vf[3][b].w}};
#pragma unroll
      for (int e = 0; e < 16; ++e) {  // independent products side by side
        const int j = e & 7;
        const uint32_t sel = (j & 1) ? 0x7632u : 0x5410u;
        mma_16816(acc[b][j], a0, e < 8 ? a1 : c1, a2, e < 8 ? a3 : c3, __byte_perm(w[0][j >> 1], w[1][j >> 1], sel),
                  __byte_perm(w[2][j >> 1], w[3][j >> 1], sel));
      }
    }
  }
  l += __shfl_xor_sync(0xffffffffu, l, 1);
  l += __shfl_xor_sync(0xffffffffu, l, 2);
  if (r < ng) {
    if (c == 0) {
      wm[warp][r] = m;
      wl[warp][r] = l;
    }
#pragma unroll
    for (int b = 0; b < VB; ++b)
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        // an infinite V times a zero term is NaN: the others count where the first is finite
        const float x0 = acc[b][j][0], x1 = acc[b][j][1];
        wo[warp][r][64 * b + 16 * c + j] = isfinite(x0) ? x0 + acc[b][j][2] : x0;
        wo[warp][r][64 * b + 16 * c + 8 + j] = isfinite(x1) ? x1 + acc[b][j][3] : x1;
      }
  }
  __syncthreads();
  // merge of states (m_i, l_i, o_i): m = max m_i, l = sum l_i 2^(m_i - m), o = sum o_i 2^(m_i - m)
  // (a state without keys has m = -inf and contributes nothing)
  for (int e = threadIdx.x; e < ng * HD; e += kDecWarps * 32) {
    const int h = e / HD, d = e - h * HD;
    float mt = -INFINITY;
#pragma unroll
    for (int w = 0; w < kDecWarps; ++w) mt = fmaxf(mt, wm[w][h]);
    float lt = 0.0f, ot = 0.0f;
#pragma unroll
    for (int w = 0; w < kDecWarps; ++w) {
      const float f = wm[w][h] == -INFINITY ? 0.0f : exp2f(wm[w][h] - mt);
      lt = fmaf(wl[w][h], f, lt);
      ot = fmaf(wo[w][h][d], f, ot);
    }
    co[h][d] = ot;
    if (d == 0) {
      cm[h] = mt;
      cl[h] = lt;
    }
  }
  cluster.sync();
  const int e1 = (rank + 1) * ng * HD / S;
  for (int e = rank * ng * HD / S + int(threadIdx.x); e < e1; e += kDecWarps * 32) {
    const int h = e / HD, d = e - h * HD;
    float ms[kDecMaxSplit], ls[kDecMaxSplit], os[kDecMaxSplit];  // every CTA's state, loads in flight
#pragma unroll
    for (int k = 0; k < kDecMaxSplit; ++k) {
      ms[k] = -INFINITY;
      ls[k] = os[k] = 0.0f;
      if (k < S) {
        ms[k] = *cluster.map_shared_rank(&cm[h], k);
        ls[k] = *cluster.map_shared_rank(&cl[h], k);
        os[k] = *cluster.map_shared_rank(&co[h][d], k);
      }
    }
    float mt = -INFINITY;
#pragma unroll
    for (int k = 0; k < kDecMaxSplit; ++k) mt = fmaxf(mt, ms[k]);
    float lt = 0.0f, ot = 0.0f;
#pragma unroll
    for (int k = 0; k < kDecMaxSplit; ++k) {
      const float f = ms[k] == -INFINITY ? 0.0f : exp2f(ms[k] - mt);
      lt = fmaf(ls[k], f, lt);
      ot = fmaf(os[k], f, ot);
    }
    o[size_t(tl.x) * ldo + (h0 + h) * HD + d] = __float2bfloat16_rn(ot / lt);
  }
  cluster.sync();  // the peers' shared memory stays alive until every CTA has read it
  if (threadIdx.x == 0) stamp_end(stamp);
}

}  // namespace

int attention_run(const void* q, int n_q, const void* kv, int n_kv, int ldkv, int v_off, void* o,
                  int ldo, const int4* tiles, int n_tiles, const int32_t* q_pos, int n_heads,
                  int n_kv_heads, int head_dim, int* status, cudaStream_t stream, double ctx_sum) {
  if (n_tiles <= 0) return SPD_OK;
  if (head_dim != 128 && head_dim != 64)
    return fail(SPD_EUNSUPPORTED, "attention supports head_dim 64 and 128");
  if (n_kv_heads < 1 || n_heads % n_kv_heads)
    return fail(SPD_EINVAL, "n_heads must be a multiple of n_kv_heads");
  if (v_off % 64 || ldkv < v_off + n_kv_heads * head_dim)
    return fail(SPD_EINVAL, "V must start at a multiple of 64 columns inside each K/V row");
  CUtensorMap mq, mkv;
  if (int rc = make_operand_map(&mq, q, n_heads * head_dim, n_q, 128)) return rc;
  if (int rc = make_operand_map(&mkv, kv, ldkv, n_kv, kTK)) return rc;
  // QK^T and PV over each active query's causal context; Q, K, V read once and O written once
  const double fl = 4.0 * head_dim * n_heads * ctx_sum;
  const double by = 2.0 * (2.0 * n_q * n_heads * head_dim + 2.0 * n_kv * n_kv_heads * head_dim);
  unsigned long long* stamp = stamp_slot(TR_ATTN, fl, by);
  const int slot = trace_begin(stream);
  const int rc = (head_dim == 128)
                     ? launch<128>(mq, mkv, o, ldo, tiles, n_tiles, q_pos, n_heads, n_kv_heads,
                                   v_off, status, stream, stamp)
                     : launch<64>(mq, mkv, o, ldo, tiles, n_tiles, q_pos, n_heads, n_kv_heads,
                                  v_off, status, stream, stamp);
  trace_end(slot, stream, TR_ATTN, fl, by);
  return rc;
}

int attention_decode_run(const void* q, const void* kv, int ldkv, int v_off, void* o, int ldo,
                         const int4* tiles, int n_tiles, int n_heads, int n_kv_heads, int head_dim,
                         cudaStream_t stream, double ctx_sum) {
  if (n_tiles <= 0) return SPD_OK;
  if (head_dim != 128 && head_dim != 64)
    return fail(SPD_EUNSUPPORTED, "attention supports head_dim 64 and 128");
  if (n_kv_heads < 1 || n_heads % n_kv_heads)
    return fail(SPD_EINVAL, "n_heads must be a multiple of n_kv_heads");
  if ((ldkv | v_off) % 4) return fail(SPD_EINVAL, "K/V rows must be 8-byte aligned");
  const float scale_log2 = float(1.4426950408889634 / sqrt(double(head_dim)));
  // Q read and O written once per query; K and V of every visible key once per KV head
  const double fl = 4.0 * head_dim * n_heads * ctx_sum;
  const double by = 2.0 * (2.0 * n_tiles * n_heads * head_dim + 2.0 * ctx_sum * n_kv_heads * head_dim);
  unsigned long long* stamp = stamp_slot(TR_ATTN, fl, by);
  const int slot = trace_begin(stream);
  const auto* qb = static_cast<const __nv_bfloat16*>(q);
  const auto* kb = static_cast<const __nv_bfloat16*>(kv);
  auto* ob = static_cast<__nv_bfloat16*>(o);
  const int chunks = (n_heads / n_kv_heads + kDecHeads - 1) / kDecHeads;
  // CTAs a sequence: more of them while two CTAs an SM are not reached and each still has 64 keys on
  // average. Measured, us a decode step, S = 1 / 2 / 4 / 8: 32 sequences of 1122 keys on average, 4 K/V
  // heads, 4 layers 894 / 829 / 858 / 976; one sequence of 257 keys, 32 K/V heads, 32 layers - / 3174 /
  // 3142 / 3395; one of 1900 keys, 4 layers 612 / 539 / 502 / 495.
  const long long groups = (long long)n_tiles * n_kv_heads * chunks;
  int S = 1;
  while (S < kDecMaxSplit && groups * 2 * S <= 2LL * num_sms() && ctx_sum >= 128.0 * S * n_tiles) S *= 2;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(n_tiles * n_kv_heads * chunks, 1, S);
  cfg.blockDim = dim3(kDecWarps * 32);
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = 1;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = S;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  const bool a16 = (reinterpret_cast<uintptr_t>(kv) & 15) == 0 && (ldkv | v_off) % 8 == 0;
  auto kern = head_dim == 128 ? (a16 ? attn_decode_kernel<128, true> : attn_decode_kernel<128, false>)
                              : (a16 ? attn_decode_kernel<64, true> : attn_decode_kernel<64, false>);
  SPD_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, qb, kb, ldkv, v_off, ob, ldo, tiles, n_heads, n_kv_heads, chunks,
                                  scale_log2, stamp));
  trace_end(slot, stream, TR_ATTN, fl, by);
  return SPD_OK;
}

}  // namespace spd
