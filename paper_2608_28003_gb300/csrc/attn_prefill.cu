// Prefill attention (many new tokens per sequence) on the 5th-generation tensor cores.
//
// Two kernels a layer.  prefill_rope_kernel turns the q/k/v projection's rows into the operands: q
// after QK-norm and RoPE, scaled and rounded to fp16; k (after QK-norm and RoPE) and v into the
// bf16 cache and, as fp16, into this layer's operand scratch: K [keys][256] and V transposed
// [256][keys], so that both products read K-major tiles.  (fp16, not bf16: 11 mantissa bits keep scores
// and probabilities close to the fp32 arithmetic of the other paths; a cached bf16 value in fp16's
// normal range is exact.)  Keys of earlier calls are converted from the cache.
//
// attn_prefill_kernel: a CTA takes 128 queries of one head and walks the keys in tiles of 128:
//  * warp 4 copies by TMA: the queries once (64 KB), then a K and a V tile (64 KB each) per step, each
//    refilled as soon as the MMAs that read it have completed; warp 5 allocates tensor memory and
//    issues tcgen05.mma: S = Q K^T (128 x 128 x 256) into one of two 128-column slots, and O += P V
//    (128 x 256 x 128) into 256 columns.  S of the next tile is issued before P of this one is awaited,
//    so the tensor cores work while the softmax runs;
//  * warps 0-3: thread = query row (its TMEM lane).  It reads its 128 scores, masks them (causal,
//    sliding window), takes the row maximum, p = exp(s - m), adds to the row sum (fp32) and writes P as
//    fp16 into the swizzled shared-memory tile the second product reads.  m only moves when the
//    maximum grew by more than 5.5 (p stays below e^5.5 = 245): O is then rescaled in tensor
//    memory, rarely after the first tiles (the conditional rescaling that FlashAttention-4 published); any m
//    gives the same quotient O / l;
//  * a call with few tiles leaves most of the SMs idle, so the key tiles of a query block are split over the
//    two CTAs of a cluster (tiles r, r + 2, ...), which exchange (m, l) and half of their O through
//    distributed shared memory and finish 128 output dims each.
// What bounds it at 2048 tokens: per tile 2048 cycles of MMA at the nominal rate beside about 1600 of
// softmax (128 exponentials per thread at 1/8 rate), 5-8 tiles per CTA, plus the ramp and the
// merge: 21 us a layer with the 1024-token window and 28 us a global one, against 70 and 118 us
// of mma.sync on 64-query blocks before (2048-token prefill with all logits 5.66 -> 4.25 ms).
// Every wait is bounded: on timeout the kernel sets a bit of the error word, stops issuing, and still
// passes its cluster barriers and frees its tensor memory.
#include <cmath>

#include "decoder_kernels.cuh"
#include "tc_common.cuh"
#include "tmap.cuh"

namespace w8a8 {

namespace {

constexpr int kHd = 256;
constexpr int kTok = 32;                  // tokens per block of the rope kernel
constexpr int kBq = 128, kBk = 128;       // queries per CTA, keys per tile
constexpr int kSub = 128 * 128;           // bytes of a 128-row sub-tile of 64 fp16 columns
constexpr uint32_t kQBytes = 4 * kSub, kKBytes = 4 * kSub, kVBytes = 4 * kSub, kPBytes = 2 * kSub;
constexpr int kOffQ = 0, kOffK = kOffQ + kQBytes, kOffV = kOffK + kKBytes, kOffP = kOffV + kVBytes;
constexpr int kAttnSmem = kOffP + kPBytes + 1024;  // 224 KB of tiles
constexpr int kSoftWarps = 4, kLoadWarp = 4, kIssueWarp = 5, kThreads = 192;
constexpr uint32_t kSCol = 0, kOCol = 256;  // tensor memory: two S slots of 128 columns, O
constexpr float kMaxGrowth = 5.5f;

__device__ __forceinline__ uint32_t pack_f16(float a, float b) {  // a in the low half
  uint32_t r;
  asm("cvt.rn.f16x2.f32 %0, %1, %2;\n" : "=r"(r) : "f"(b), "f"(a));
  return r;
}
__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;\n" : "=r"(r) : "f"(b), "f"(a));
  return r;
}
__device__ __forceinline__ uint32_t bf16x2_to_f16x2(uint32_t w) { return pack_f16(bf16_lo(w), bf16_hi(w)); }

// ---------------------------------------------------------------------------- operands
// grid (token blocks of 32: the call's tokens padded to a key multiple of 128, then the keys of
// earlier calls; heads: q, k, v; sequences), 8 warps of 4 tokens.  Lane l of a warp holds dims
// 4l .. 4l+3 and 128 + 4l .. 128 + 4l + 3 of its token: the four RoPE pairs (i, i + 128).
// Latency bounds it (12 MB at 2048 tokens, 2 us of copy): the RoPE factors are read ahead of the wait for the
// projection and the four tokens' rows before the first is used: 8.0 -> 6.7 us a launch at 2048 tokens.
__global__ void __launch_bounds__(256) prefill_rope_kernel(const uint16_t* __restrict__ qkv, AttnShape s, int p0,
                                                           const float* __restrict__ qn, const float* __restrict__ kn,
                                                           float eps, const float* __restrict__ rope_cos,
                                                           const float* __restrict__ rope_sin, uint16_t* __restrict__ q16,
                                                           uint16_t* __restrict__ kcache, uint16_t* __restrict__ vcache,
                                                           uint16_t* __restrict__ k16, uint16_t* __restrict__ vt,
                                                           int keys_pad, int new_blocks) {
  __shared__ uint16_t tile[kTok][kHd + 2];  // a V block for the transposition
  pdl_trigger();
  const int head = blockIdx.y, b = blockIdx.z;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool is_q = head < s.n_q, is_k = !is_q && head < s.n_q + s.n_kv;
  const bool fresh = (int)blockIdx.x < new_blocks;  // this call's tokens, else earlier keys
  if (!fresh && is_q) return;
  const int kvh = is_q ? 0 : is_k ? head - s.n_q : head - s.n_q - s.n_kv;
  const int key0 = fresh ? p0 + (int)blockIdx.x * kTok : ((int)blockIdx.x - new_blocks) * kTok;
  const int key_end = fresh ? p0 + s.T : p0;  // keys from here on are padding (fresh) or another block's
  const size_t row_stride = (size_t)s.n_kv * kHd;
  const size_t cache0 = (size_t)b * s.max_seq * row_stride + (size_t)kvh * kHd;
  const size_t op0 = ((size_t)b * s.n_kv + kvh) * keys_pad;  // operand scratch: first key row
  float nw1[4], nw2[4];
  const float* nw = is_q ? qn : is_k ? kn : nullptr;
  if (nw) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      nw1[e] = nw[4 * lane + e];
      nw2[e] = nw[128 + 4 * lane + e];
    }
  }
  constexpr int kPer = kTok / 8;  // tokens of a warp: the loads of all of them ahead of the first use
  float4 csr[kPer], snr[kPer];
  if (fresh && (is_q || is_k)) {
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const int key = min(key0 + warp * kPer + i, key_end - 1);
      csr[i] = *reinterpret_cast<const float4*>(rope_cos + (size_t)key * 128 + 4 * lane);
      snr[i] = *reinterpret_cast<const float4*>(rope_sin + (size_t)key * 128 + 4 * lane);
    }
  }
  pdl_wait();
  const int qkv_dim = (s.n_q + 2 * s.n_kv) * kHd;
  uint2 ar[kPer], cr[kPer];
#pragma unroll
  for (int i = 0; i < kPer; ++i) {
    const int key = key0 + warp * kPer + i;
    ar[i] = cr[i] = make_uint2(0u, 0u);
    if (key < key_end) {
      const uint16_t* src = fresh ? qkv + ((size_t)b * s.T + key - p0) * qkv_dim + (size_t)head * kHd
                                  : (is_k ? kcache : vcache) + cache0 + (size_t)key * row_stride;
      ar[i] = *reinterpret_cast<const uint2*>(src + 4 * lane);
      cr[i] = *reinterpret_cast<const uint2*>(src + 128 + 4 * lane);
    }
  }
#pragma unroll
  for (int i = 0; i < kPer; ++i) {
    const int j = warp * kPer + i, key = key0 + j;
    const bool live = key < key_end;
    uint2 a = ar[i], c = cr[i];
    const int t = key - p0;
    if (!is_q && !is_k) {  // v: cache as is, fp16 transposed below
      if (fresh && live) {
        uint16_t* dst = vcache + cache0 + (size_t)key * row_stride;
        *reinterpret_cast<uint2*>(dst + 4 * lane) = a;
        *reinterpret_cast<uint2*>(dst + 128 + 4 * lane) = c;
      }
      uint32_t* r = reinterpret_cast<uint32_t*>(&tile[j][0]);
      r[2 * lane] = bf16x2_to_f16x2(a.x);
      r[2 * lane + 1] = bf16x2_to_f16x2(a.y);
      r[64 + 2 * lane] = bf16x2_to_f16x2(c.x);
      r[64 + 2 * lane + 1] = bf16x2_to_f16x2(c.y);
      continue;
    }
    if (fresh && live) {
      float x1[4] = {bf16_lo(a.x), bf16_hi(a.x), bf16_lo(a.y), bf16_hi(a.y)};
      float x2[4] = {bf16_lo(c.x), bf16_hi(c.x), bf16_lo(c.y), bf16_hi(c.y)};
      if (nw) {
        float ss = 0.0f;
#pragma unroll
        for (int e = 0; e < 4; ++e) ss += x1[e] * x1[e] + x2[e] * x2[e];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
        const float inv = 1.0f / sqrtf(ss / (float)kHd + eps);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          x1[e] = x1[e] * inv * nw1[e];
          x2[e] = x2[e] * inv * nw2[e];
        }
      }
      const float4 cs = csr[i], sn = snr[i];
      const float cv[4] = {cs.x, cs.y, cs.z, cs.w}, sv[4] = {sn.x, sn.y, sn.z, sn.w};
      float y1[4], y2[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        y1[e] = x1[e] * cv[e] - x2[e] * sv[e];
        y2[e] = x2[e] * cv[e] + x1[e] * sv[e];
      }
      if (is_q) {
        uint16_t* dst = q16 + ((size_t)b * s.T + t) * (s.n_q * kHd) + (size_t)head * kHd;
        *reinterpret_cast<uint2*>(dst + 4 * lane) =
            make_uint2(pack_f16(y1[0] * s.scale, y1[1] * s.scale), pack_f16(y1[2] * s.scale, y1[3] * s.scale));
        *reinterpret_cast<uint2*>(dst + 128 + 4 * lane) =
            make_uint2(pack_f16(y2[0] * s.scale, y2[1] * s.scale), pack_f16(y2[2] * s.scale, y2[3] * s.scale));
        continue;
      }
      a = make_uint2(pack_bf16(y1[0], y1[1]), pack_bf16(y1[2], y1[3]));
      c = make_uint2(pack_bf16(y2[0], y2[1]), pack_bf16(y2[2], y2[3]));
      uint16_t* dst = kcache + cache0 + (size_t)key * row_stride;
      *reinterpret_cast<uint2*>(dst + 4 * lane) = a;
      *reinterpret_cast<uint2*>(dst + 128 + 4 * lane) = c;
    }
    if (is_k && key < keys_pad && (live || fresh)) {  // the cached (bf16) value as fp16; zeros in the padding
      uint16_t* dst = k16 + (op0 + key) * kHd;
      *reinterpret_cast<uint2*>(dst + 4 * lane) = make_uint2(bf16x2_to_f16x2(a.x), bf16x2_to_f16x2(a.y));
      *reinterpret_cast<uint2*>(dst + 128 + 4 * lane) = make_uint2(bf16x2_to_f16x2(c.x), bf16x2_to_f16x2(c.y));
    }
  }
  if (is_q || is_k) return;
  __syncthreads();
  const int key = key0 + lane;
  if (key < keys_pad && (key < key_end || fresh)) {
    uint16_t* dst = vt + ((size_t)b * s.n_kv + kvh) * kHd * keys_pad + key;
#pragma unroll 8
    for (int i = 0; i < kHd / 8; ++i) {
      const int d = warp * (kHd / 8) + i;
      dst[(size_t)d * keys_pad] = tile[lane][d];
    }
  }
}

// -------------------------------------------------------------------------- attention
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}
__device__ __forceinline__ uint32_t map_to_rank(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ float exp_of(float x) {  // e^x, x <= 5.5 or -inf
  float r;
  asm("ex2.approx.ftz.f32 %0, %1;\n" : "=f"(r) : "f"(x * 1.4426950408889634f));
  return r;
}
// 32 values into 32 consecutive tensor-memory columns of this thread's lane
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%32], {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31};\n" ::"r"(r[0]),
      "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]),
      "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]),
      "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]),
      "r"(r[29]), "r"(r[30]), "r"(r[31]), "r"(taddr)
      : "memory");
}

template <int kSplit>
__global__ void __cluster_dims__(kSplit, 1, 1) __launch_bounds__(kThreads, 1)
    attn_prefill_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                        const __grid_constant__ CUtensorMap tmV, AttnShape s, int p0, int keys_pad,
                        uint16_t* __restrict__ o, unsigned int* __restrict__ err) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  enum { Q_FULL, K_FULL, K_FREE, V_FULL, V_FREE, S_FULL0, S_FULL1, S_FREE0, S_FREE1, P_FULL, PV_DONE, ALL_DONE, N_BARS };
  __shared__ uint64_t bars[N_BARS];
  __shared__ uint32_t tmem_slot;
  __shared__ float2 s_ml[kSplit > 1 ? kBq : 1];  // (m, l) of the peer's rows

  const uint32_t raw = smem_u32(smem_raw), base = (raw + 1023u) & ~1023u;
  const uint32_t bar0 = smem_u32(bars);
  auto bar = [&](int i) { return bar0 + 8u * (uint32_t)i; };
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = kSplit > 1 ? cluster_rank() : 0u;
  const int qb = blockIdx.x / kSplit, head = blockIdx.y, b = blockIdx.z;
  const int kvh = head / (s.n_q / s.n_kv);
  const int t0 = qb * kBq, t_last = min(s.T, t0 + kBq) - 1;
  const int hi = p0 + t_last;                                           // last key any query of the block sees
  const int lo = s.window > 0 ? max(0, p0 + t0 - s.window + 1) : 0;     // first one
  const int tile0 = lo / kBk + (int)rank;                               // this CTA's tiles: tile0, tile0 + kSplit, ...
  const int n = tile0 <= hi / kBk ? (hi / kBk - tile0) / kSplit + 1 : 0;

  pdl_trigger();
  if (threadIdx.x == 0) {
    for (int i = 0; i < N_BARS; ++i) mbar_init(bar(i), i == S_FREE0 || i == S_FREE1 || i == P_FULL ? kBq : 1);
    fence_mbar_init();
    prefetch_tmap(&tmQ);
    prefetch_tmap(&tmK);
    prefetch_tmap(&tmV);
  }
  if (warp == kIssueWarp) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;\n" ::"r"(smem_u32(&tmem_slot))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  if constexpr (kSplit > 1) cluster_sync_all();  // the peer runs: its shared memory may be written
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  pdl_wait();

  float m = -INFINITY, l = 0.0f;  // softmax threads: this row's reference and sum
  bool ok = true;
  if (warp == kLoadWarp) {
    // ------------------------------------------------------------------------ TMA copies
    const int krow = (b * s.n_kv + kvh) * keys_pad, vrow = (b * s.n_kv + kvh) * kHd;
    if (n > 0) {
      if (elect_one()) {
        mbar_arrive_expect_tx(bar(Q_FULL), kQBytes);
#pragma unroll
        for (int c = 0; c < 4; ++c)
          tma_load_2d(base + kOffQ + c * kSub, &tmQ, head * kHd + 64 * c, b * s.T + t0, bar(Q_FULL));
      }
      __syncwarp();
      int nk = 0, nv = 0;  // copies issued
      for (int i = 0; i < n; ++i) {
        const int j0 = (tile0 + kSplit * i) * kBk;
        const uint32_t ph = (uint32_t)((i & 1) ^ 1);
        if (!mbar_wait_warp(bar(K_FREE), ph, kWaitBudgetCycles)) {
          ok = false;
          break;
        }
        if (elect_one()) {
          mbar_arrive_expect_tx(bar(K_FULL), kKBytes);
#pragma unroll
          for (int c = 0; c < 4; ++c) tma_load_2d(base + kOffK + c * kSub, &tmK, 64 * c, krow + j0, bar(K_FULL));
        }
        __syncwarp();
        ++nk;
        if (!mbar_wait_warp(bar(V_FREE), ph, kWaitBudgetCycles)) {
          ok = false;
          break;
        }
        if (elect_one()) {
          mbar_arrive_expect_tx(bar(V_FULL), kVBytes);
#pragma unroll
          for (int c = 0; c < 2; ++c) tma_load_2d(base + kOffV + c * 2 * kSub, &tmV, j0 + 64 * c, vrow, bar(V_FULL));
        }
        __syncwarp();
        ++nv;
      }
      if (lane == 0) {
        if (!ok) atomicOr(err, DEVERR_PRODUCER_WAIT);
        // the last copies land before the tiles are used for anything else
        if (!mbar_wait_bounded(bar(Q_FULL), 0u, kWaitBudgetCycles) ||
            (nk > 0 && !mbar_wait_bounded(bar(K_FULL), (uint32_t)(nk - 1) & 1u, kWaitBudgetCycles)) ||
            (nv > 0 && !mbar_wait_bounded(bar(V_FULL), (uint32_t)(nv - 1) & 1u, kWaitBudgetCycles)))
          atomicOr(err, DEVERR_DRAIN_WAIT);
      }
      __syncwarp();
    }
  } else if (warp == kIssueWarp) {
    // ------------------------------------------------------------------------ MMAs
    constexpr uint32_t idesc_s = idesc_f16(0u, kBk, kBq), idesc_o = idesc_f16(0u, kHd, kBq);
    const uint64_t dq = sdesc_swz(base + kOffQ), dk = sdesc_swz(base + kOffK), dv = sdesc_swz(base + kOffV),
                   dp = sdesc_swz(base + kOffP);
    auto issue_s = [&](int i) {  // S_i = Q K_i^T
      if (!mbar_wait_warp(bar(K_FULL), (uint32_t)(i & 1), kWaitBudgetCycles)) return false;
      if (i >= 2 && !mbar_wait_warp(bar(S_FREE0 + (i & 1)), (uint32_t)((i >> 1) - 1) & 1u, kWaitBudgetCycles)) return false;
      tc_fence_after();
      if (elect_one()) {
        const uint32_t d = tmem + kSCol + 128u * (uint32_t)(i & 1);
#pragma unroll
        for (int k = 0; k < kHd / 16; ++k) {
          const uint32_t at = (uint32_t)((k >> 2) * (kSub >> 4) + 2 * (k & 3));
          tc_mma(d, dq + at, dk + at, idesc_s, k > 0);
        }
        tc_commit(bar(K_FREE));
        tc_commit(bar(S_FULL0 + (i & 1)));
      }
      __syncwarp();
      return true;
    };
    if (n > 0) {
      ok = mbar_wait_warp(bar(Q_FULL), 0u, kWaitBudgetCycles) && issue_s(0);
      for (int i = 0; i < n && ok; ++i) {
        if (i + 1 < n && !issue_s(i + 1)) {
          ok = false;
          break;
        }
        if (!mbar_wait_warp(bar(V_FULL), (uint32_t)(i & 1), kWaitBudgetCycles) ||
            !mbar_wait_warp(bar(P_FULL), (uint32_t)(i & 1), kWaitBudgetCycles)) {
          ok = false;
          break;
        }
        tc_fence_after();
        if (elect_one()) {  // O += P_i V_i
#pragma unroll
          for (int k = 0; k < kBk / 16; ++k)
            tc_mma(tmem + kOCol, dp + (uint32_t)((k >> 2) * (kSub >> 4) + 2 * (k & 3)),
                   dv + (uint32_t)((k >> 2) * (2 * kSub >> 4) + 2 * (k & 3)), idesc_o, i > 0 || k > 0);
          tc_commit(bar(V_FREE));
          tc_commit(bar(PV_DONE));
        }
        __syncwarp();
      }
      if (elect_one()) {
        if (!ok) atomicOr(err, DEVERR_PRODUCER_WAIT);
        tc_commit(bar(ALL_DONE));  // completes once every MMA issued above has
        if (!mbar_wait_bounded(bar(ALL_DONE), 0u, kWaitBudgetCycles)) atomicOr(err, DEVERR_DRAIN_WAIT);
      }
      __syncwarp();
    }
  } else {
    // ------------------------------------------------------------------------ softmax, one row per thread
    const int r = threadIdx.x;                             // query row of the block, TMEM lane
    const int p = p0 + t0 + r;                             // its position (rows past the call's tokens are not stored)
    const int row_lo = s.window > 0 ? max(0, p - s.window + 1) : 0;
    const uint32_t lanes = tmem + ((uint32_t)(32 * warp) << 16);
    const uint32_t prow = base + kOffP + (uint32_t)(r * 128);
    for (int i = 0; i < n; ++i) {
      const int j0 = (tile0 + kSplit * i) * kBk;
      if (!mbar_wait_warp(bar(S_FULL0 + (i & 1)), (uint32_t)(i >> 1) & 1u, kWaitBudgetCycles)) {
        ok = false;
        break;
      }
      tc_fence_after();
      float v[kBk];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        uint32_t w[32];
        tmem_ld32(lanes + kSCol + 128u * (uint32_t)(i & 1) + 32 * c, w);
#pragma unroll
        for (int k = 0; k < 32; ++k) v[32 * c + k] = __uint_as_float(w[k]);
      }
      tc_fence_before();
      mbar_arrive(bar(S_FREE0 + (i & 1)));
      if (j0 < row_lo || j0 + kBk - 1 > p) {
#pragma unroll
        for (int k = 0; k < kBk; ++k)
          if (j0 + k < row_lo || j0 + k > p) v[k] = -INFINITY;
      }
      float mx[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) mx[k] = v[k];
#pragma unroll
      for (int k = 8; k < kBk; ++k) mx[k & 7] = fmaxf(mx[k & 7], v[k]);
      const float top = fmaxf(fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])), fmaxf(fmaxf(mx[4], mx[5]), fmaxf(mx[6], mx[7])));
      float scale = 1.0f;
      const bool grown = top > m + kMaxGrowth;  // m = -inf: any visible key
      if (grown) {
        scale = m == -INFINITY ? 0.0f : exp_of(m - top);
        m = top;
        l *= scale;
      }
      const float mref = m == -INFINITY ? 0.0f : m;  // no visible key yet: every p is 0
      float sum[4] = {0.0f, 0.0f, 0.0f, 0.0f};
      uint32_t pk[kBk / 2];
#pragma unroll
      for (int k = 0; k < kBk; k += 2) {
        const float e0 = exp_of(v[k] - mref), e1 = exp_of(v[k + 1] - mref);
        sum[(k >> 1) & 3] += e0 + e1;
        pk[k >> 1] = pack_f16(e0, e1);
      }
      l += (sum[0] + sum[1]) + (sum[2] + sum[3]);
      // the P tile and O are free once the previous tile's product has completed
      if (i > 0 && !mbar_wait_warp(bar(PV_DONE), (uint32_t)(i - 1) & 1u, kWaitBudgetCycles)) {
        ok = false;
        break;
      }
      if (i > 0 && __any_sync(0xffffffffu, grown)) {
        tc_fence_after();
#pragma unroll 1
        for (int c = 0; c < kHd / 32; ++c) {
          uint32_t w[32];
          tmem_ld32(lanes + kOCol + 32 * c, w);
#pragma unroll
          for (int k = 0; k < 32; ++k) w[k] = __float_as_uint(__uint_as_float(w[k]) * scale);
          tmem_st32(lanes + kOCol + 32 * c, w);
        }
        asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory");
        tc_fence_before();
      }
#pragma unroll
      for (int c = 0; c < kBk / 8; ++c)
        asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};\n" ::"r"(prow + (uint32_t)((c >> 3) * kSub) +
                                                                        (uint32_t)(((c & 7) ^ (r & 7)) << 4)),
                     "r"(pk[4 * c]), "r"(pk[4 * c + 1]), "r"(pk[4 * c + 2]), "r"(pk[4 * c + 3])
                     : "memory");
      asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
      mbar_arrive(bar(P_FULL));
    }
    if (ok && n > 0 && !mbar_wait_warp(bar(PV_DONE), (uint32_t)(n - 1) & 1u, kWaitBudgetCycles)) ok = false;
    if (!ok && lane == 0) atomicOr(err, DEVERR_CONSUMER_WAIT);
    __syncwarp();
    tc_fence_after();
  }

  // ---------------------------------------------------------------------- output: O / l as bf16
  const bool soft = warp < kSoftWarps;
  const int r = threadIdx.x;
  const uint32_t lanes = tmem + ((uint32_t)(32 * (warp & 3)) << 16);
  const int t = t0 + r;
  uint16_t* orow = o + ((size_t)b * s.T + t) * (s.n_q * kHd) + (size_t)head * kHd;
  auto load_o = [&](int c, float f, float (&x)[32]) {  // 32 dims of this row, times f
    uint32_t w[32];
    tmem_ld32(lanes + kOCol + 32 * c, w);
#pragma unroll
    for (int k = 0; k < 32; ++k) x[k] = __uint_as_float(w[k]) * f;
  };
  auto store_o = [&](int c, const float (&x)[32]) {
    if (t >= s.T) return;
#pragma unroll
    for (int k = 0; k < 4; ++k)
      reinterpret_cast<uint4*>(orow + 32 * c)[k] =
          make_uint4(pack_bf16(x[8 * k], x[8 * k + 1]), pack_bf16(x[8 * k + 2], x[8 * k + 3]),
                     pack_bf16(x[8 * k + 4], x[8 * k + 5]), pack_bf16(x[8 * k + 6], x[8 * k + 7]));
  };
  if constexpr (kSplit == 1) {
    if (soft && n > 0) {
      const float f = l > 0.0f ? 1.0f / l : 0.0f;
#pragma unroll 1
      for (int c = 0; c < kHd / 32; ++c) {
        float x[32];
        load_o(c, f, x);
        store_o(c, x);
      }
    }
  } else {
    const uint32_t peer = rank ^ 1u;
    if (soft) {
      asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};\n" ::"r"(map_to_rank(smem_u32(s_ml + r), peer)), "f"(m),
                   "f"(l)
                   : "memory");
    }
    cluster_sync_all();  // (m, l) exchanged; both CTAs' products are complete, so the tiles are free
    float f = 0.0f;
    if (soft) {
      const float m1 = s_ml[r].x, l1 = s_ml[r].y, mm = fmaxf(m, m1);
      const float e0 = m == -INFINITY ? 0.0f : exp_of(m - mm), e1 = m1 == -INFINITY ? 0.0f : exp_of(m1 - mm);
      const float sum = l * e0 + l1 * e1;
      f = sum > 0.0f ? e0 / sum : 0.0f;
      // the peer's half of the dims: into its Q / K area, [16-byte chunk][row]
      const uint32_t dst = map_to_rank(base + kOffQ, peer) + (uint32_t)(r * 16);
#pragma unroll 1
      for (int c = 0; c < kHd / 64; ++c) {
        float x[32];
        if (n > 0)
          load_o((int)peer * (kHd / 64) + c, f, x);
        else
#pragma unroll
          for (int k = 0; k < 32; ++k) x[k] = 0.0f;
#pragma unroll
        for (int k = 0; k < 8; ++k)
          asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};\n" ::"r"(dst + (uint32_t)((8 * c + k) * kBq * 16)),
                       "f"(x[4 * k]), "f"(x[4 * k + 1]), "f"(x[4 * k + 2]), "f"(x[4 * k + 3])
                       : "memory");
      }
    }
    cluster_sync_all();
    if (soft) {
#pragma unroll 1
      for (int c = 0; c < kHd / 64; ++c) {
        float x[32];
        if (n > 0)
          load_o((int)rank * (kHd / 64) + c, f, x);
        else
#pragma unroll
          for (int k = 0; k < 32; ++k) x[k] = 0.0f;
        const float4* mine = reinterpret_cast<const float4*>(smem_raw + (base - raw) + kOffQ) + (size_t)(8 * c) * kBq + r;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const float4 y = mine[k * kBq];
          x[4 * k] += y.x;
          x[4 * k + 1] += y.y;
          x[4 * k + 2] += y.z;
          x[4 * k + 3] += y.w;
        }
        store_o((int)rank * (kHd / 64) + c, x);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kIssueWarp) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;\n" ::"r"(tmem) : "memory");
  }
}

template <int kSplit>
w8a8_status launch_split(const CUtensorMap& tq, const CUtensorMap& tk, const CUtensorMap& tv, const AttnShape& s, int pos0,
                         int keys_pad, uint16_t* o, unsigned int* err, cudaStream_t st) {
  static bool attr_set[64] = {};
  int dev = 0;
  W8A8_CUDA(cudaGetDevice(&dev));
  if (dev >= 0 && dev < 64 && !attr_set[dev]) {
    W8A8_CUDA(cudaFuncSetAttribute(attn_prefill_kernel<kSplit>, cudaFuncAttributeMaxDynamicSharedMemorySize, kAttnSmem));
    attr_set[dev] = true;
  }
  const dim3 grid((unsigned)(kSplit * ((s.T + kBq - 1) / kBq)), (unsigned)s.n_q, (unsigned)s.B);
  W8A8_CUDA(launch_pdl(attn_prefill_kernel<kSplit>, grid, dim3(kThreads), (size_t)kAttnSmem, st, tq, tk, tv, s, pos0,
                       keys_pad, o, err));
  return W8A8_OK;
}

}  // namespace

bool attention_prefill_supported(const AttnShape& s) {
  return s.hd == kHd && s.n_kv > 0 && s.n_q % s.n_kv == 0 && s.T > 1;
}

int prefill_keys_pad(int max_seq) { return (max_seq + kBk - 1) / kBk * kBk; }

w8a8_status launch_prefill_rope(const uint16_t* qkv, const AttnShape& s, int pos0, const float* qn, const float* kn,
                                float eps, const float* rope_cos, const float* rope_sin, uint16_t* kcache,
                                uint16_t* vcache, const PrefillOperands& w, cudaStream_t st) {
  if (s.B == 0 || s.T == 0) return W8A8_OK;
  W8A8_CHECK_ARG(attention_prefill_supported(s), W8A8_ERR_SHAPE, "prefill attention: head dim 256 and T > 1 only");
  const int keys_pad = prefill_keys_pad(s.max_seq), end = (pos0 + s.T + kBk - 1) / kBk * kBk;
  const int fresh = (end - pos0 + kTok - 1) / kTok, old = (pos0 + kTok - 1) / kTok;
  W8A8_CUDA(launch_pdl(prefill_rope_kernel, dim3((unsigned)(fresh + old), (unsigned)(s.n_q + 2 * s.n_kv), (unsigned)s.B),
                       dim3(256), 0, st, qkv, s, pos0, qn, kn, eps, rope_cos, rope_sin, w.q, kcache, vcache, w.k, w.vt,
                       keys_pad, fresh));
  return W8A8_OK;
}

w8a8_status launch_attention_prefill(const PrefillOperands& w, const AttnShape& s, int pos0, uint16_t* o, int sms,
                                     unsigned int* err, cudaStream_t st) {
  if (s.B == 0 || s.T == 0) return W8A8_OK;
  W8A8_CHECK_ARG(attention_prefill_supported(s), W8A8_ERR_SHAPE, "prefill attention: head dim 256 and T > 1 only");
  const int keys_pad = prefill_keys_pad(s.max_seq);
  const uint64_t qw = (uint64_t)s.n_q * kHd, kv = (uint64_t)s.B * s.n_kv;
  CUtensorMap tq, tk, tv;
  W8A8_TRY(make_tmap_2d(&tq, w.q, 2, qw, (uint64_t)s.B * s.T, qw * 2, 64, kBq, 128));
  W8A8_TRY(make_tmap_2d(&tk, w.k, 2, kHd, kv * keys_pad, kHd * 2, 64, kBk, 128));
  W8A8_TRY(make_tmap_2d(&tv, w.vt, 2, (uint64_t)keys_pad, kv * kHd, (uint64_t)keys_pad * 2, 64, kHd, 128));
  // two CTAs per query block while that leaves none of them waiting for an SM (2048 tokens: 64 blocks) and there is
  // more than one key tile to share
  const long long blocks = (long long)((s.T + kBq - 1) / kBq) * s.n_q * s.B;
  return 2 * blocks <= sms && pos0 + s.T > kBk ? launch_split<2>(tq, tk, tv, s, pos0, keys_pad, o, err, st)
                           : launch_split<1>(tq, tk, tv, s, pos0, keys_pad, o, err, st);
}

}  // namespace w8a8
