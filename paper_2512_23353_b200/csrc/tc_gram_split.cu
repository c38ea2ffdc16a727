// The token-Gram route and the sampled estimator (tc_gram.cu) for few tokens: a 128 x 128 tile of token pairs per CLUSTER of
// CTAs, which share the features.
//
// A tile is one chain of (d_in + d_out) / 64 stages, 0.2 us each: what one SM takes in.  Where there are fewer tiles than SMs
// that chain is all there is to wait for while most of the chip is idle (169 tokens, 3584 + 10752 features: 3 tiles, 224 stages,
// 52 us).  Here CTA r of a cluster of C takes a C-th of the stages, X's and then dY's, and ends with partial sums of P, of Q, or
// of both in its tensor memory.  P and Q have to be complete before they are multiplied: the CTAs send each other the 32 x 32
// blocks of their sums through distributed shared memory, block b to CTA b mod C, where one warp adds them in rank order and
// goes on as the other kernels' epilogues do (tc_gram_epilogue.cuh).
//
// Several projections that share X run as units of their own (P is formed once per projection: there are SMs to spare).
//
//   warp 0      TMA producer: [128 tokens] x [64 features] boxes, 4-stage ring
//   warp 1      MMA issuer: tcgen05.mma 128 x 128 x 16, K-major operands
//   warps 2-9   tensor memory -> the cluster's shared memory (a warp takes 32 rows and half of the columns); then the first
//               16 / C of them: sums, product, segmented sums, float atomics into K
#include <algorithm>

#include "tc_common.cuh"
#include "tc_gram_epilogue.cuh"

namespace isopo {

namespace {

using namespace tc;

constexpr int kTT = 128;  // tokens per tile
constexpr int kKF = 64;   // features per stage (128 bytes of bf16)
constexpr int kStages = 4;
constexpr int kOperandBytes = kTT * 128;
constexpr int kStageBytes = 2 * kOperandBytes;
constexpr int kBlockBytes = 32 * 32 * 4;
constexpr int kBlocks = 16;  // 32 x 32 blocks of a tile
constexpr int kThreads = 320;
constexpr uint32_t kTmemCols = 256;  // P 128 + Q 128
constexpr int kMaxProj = 3;
// Sums that meet in a CTA: one from every CTA for each of its blocks, and a second one from the CTA whose stages are of both.
constexpr int split_smem(int c) { return kStages * kStageBytes + (c + 1) * (kBlocks / c) * kBlockBytes + 1024 + 128; }
static_assert(split_smem(2) <= 227 * 1024, "shared memory");

struct GramSplitParams {
  const int32_t* tokseq;
  float* K[kMaxProj];  // Gram: K [B, B];  sampled: M^T [samples, B]
  int64_t T;
  int B, nT, d_in;
  int d_out[kMaxProj];
  int32_t* info;
  int n_rows, n_row_tiles;  // sampled: sample rows and their 128-row tiles
  uint32_t row_bytes;       // sampled: of a stage's row operand
  int units;                // tiles of a projection
  bool complete;            // one cluster: it fills K's other triangle as well
};

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void st_cluster_4(uint32_t cluster_addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(cluster_addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}

template <bool kSampled, int kC>
__global__ void __cluster_dims__(kC, 1, 1) __launch_bounds__(kThreads, 1)
k_bf16_gram_split(const __grid_constant__ CUtensorMap mapRX, const __grid_constant__ CUtensorMap mapRY,
                  const __grid_constant__ CUtensorMap mapX, const __grid_constant__ CUtensorMap mapY0,
                  const __grid_constant__ CUtensorMap mapY1, const __grid_constant__ CUtensorMap mapY2, GramSplitParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t smem_base = smem_u32(smem);
  constexpr int kPerCta = kBlocks / kC;  // blocks that a CTA completes
  constexpr int kSumsBytes = (kC + 1) * kPerCta * kBlockBytes;
  uint8_t* sums = smem + kStages * kStageBytes;  // [slot][block of this CTA][8][32 lanes][4 columns]
  uint64_t* bars = reinterpret_cast<uint64_t*>(sums + kSumsBytes);
  const uint32_t bar0 = smem_u32(bars);
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (kStages + s); };
  const uint32_t accfull_bar = bar0 + 8u * (2 * kStages);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kStages + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)cluster_ctarank();
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
    mbar_init(accfull_bar, 1);
    *abort_flag = 0;
    fence_barrier_init();
  }
  if (warp == 1) tmem_alloc(smem_u32(tmem_slot), kTmemCols);
  pdl_begin();
  tc_fence_before_sync();
  __syncthreads();
  cluster_arrive();  // waited for before the first store to another CTA: it has started by then
  tc_fence_after_sync();
  const uint32_t tmem_base = *tmem_slot;

  // this cluster's projection and tile
  const int cluster = blockIdx.x / kC, h = cluster / p.units;
  int u = cluster - h * p.units, I, J;
  if (kSampled) {
    I = u % p.n_row_tiles;
    J = u / p.n_row_tiles;
  } else {
    for (I = 0; u >= p.nT - I; ++I) u -= p.nT - I;  // row I holds nT - I pairs I <= J
    J = I + u;
  }
  const bool diag = !kSampled && I == J;
  const int d_out = h == 0 ? p.d_out[0] : (h == 1 ? p.d_out[1] : p.d_out[2]);
  const int nkx = (p.d_in + kKF - 1) / kKF, total = nkx + (d_out + kKF - 1) / kKF;
  auto first_of = [&](int r) { return (int)((long long)total * r / kC); };  // no share is empty: total >= C
  const int s0 = first_of(rank), s1 = first_of(rank + 1);

  if (warp == 0) {
    if (elect_one()) {
      const CUtensorMap* mapY = h == 0 ? &mapY0 : (h == 1 ? &mapY1 : &mapY2);
      int stage = 0;
      uint32_t phase = 0;
      for (int kb = s0; kb < s1; ++kb) {
        if (!mbar_wait(empty_bar(stage), phase ^ 1u, abort_flag, p.info, kIdGram)) break;
        const bool second = kb >= nkx;
        const CUtensorMap* cmap = second ? mapY : &mapX;
        const CUtensorMap* rmap = kSampled ? (second ? &mapRY : &mapRX) : cmap;
        const int x = (second ? kb - nkx : kb) * kKF;
        const uint32_t dst = smem_base + stage * kStageBytes;
        mbar_arrive_expect_tx(full_bar(stage), kSampled ? p.row_bytes + kOperandBytes : diag ? kOperandBytes : kStageBytes);
        tma_load_2d(dst, rmap, x, I * kTT, full_bar(stage));
        if (!diag) tma_load_2d(dst + kOperandBytes, cmap, x, J * kTT, full_bar(stage));
        if (++stage == kStages) { stage = 0; phase ^= 1u; }
      }
    }
    __syncwarp();
    cluster_wait();
  } else if (warp == 1) {
    if (elect_one()) {  // elected, not "lane 0": lets the compiler keep the MMA operands in uniform registers
      constexpr uint32_t idesc = make_idesc_bf16(kTT, kTT, false, false);
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      for (int kb = s0; kb < s1; ++kb) {
        if (!(ok = mbar_wait(full_bar(stage), phase, abort_flag, p.info, kIdGram))) break;
        tc_fence_after_sync();
        const uint32_t a_addr = smem_base + stage * kStageBytes;
        const uint32_t b_addr = diag ? a_addr : a_addr + kOperandBytes;
        const uint32_t d_tmem = tmem_base + (kb >= nkx ? 128u : 0u);
        const bool first = kb == s0 || kb == nkx;
#pragma unroll
        for (int k16 = 0; k16 < kKF / 16; ++k16)
          mma_bf16(d_tmem, make_sdesc_sw128(a_addr + k16 * 32, 16, 1024), make_sdesc_sw128(b_addr + k16 * 32, 16, 1024), idesc,
                   !first || k16 != 0);
        mma_commit(empty_bar(stage));
        if (++stage == kStages) { stage = 0; phase ^= 1u; }
      }
      if (ok) mma_commit(accfull_bar);
    }
    __syncwarp();
    cluster_wait();
  } else {
    const int q = warp & 3, g0 = (warp - 2) / 4 * 2;  // TMEM lanes that this warp can read; its column groups
    const bool ok = mbar_wait(accfull_bar, 0, abort_flag, p.info, kIdGram);
    tc_fence_after_sync();
    cluster_wait();
    if (ok) {
#pragma unroll 1
      for (int k = 0; k < 4; ++k) {  // P of the warp's two column groups, then Q
        const bool second = k >= 2;
        if (second ? s1 <= nkx : s0 >= nkx) continue;
        const int g = g0 + (k & 1), blk = g * 4 + q, slot = second && s0 < nkx ? kC : rank;
        uint32_t v[32];
        tmem_ld32(tmem_base + ((uint32_t)(q * 32) << 16) + (second ? 128u : 0u) + g * 32, v);
        const uint32_t to = map_to_cta(smem_u32(sums) + (uint32_t)((slot * kPerCta + blk / kC) * kBlockBytes + lane * 16), blk % kC);
        tmem_ld_wait();
#pragma unroll
        for (int e = 0; e < 8; ++e) st_cluster_4(to + e * 512, v[4 * e], v[4 * e + 1], v[4 * e + 2], v[4 * e + 3]);
      }
    }
  }
  __syncwarp();
  cluster_arrive();
  // the sequences that the sums below belong to, loaded under the barrier
  const int mine = warp - 2, blk = rank + kC * mine, g = blk >> 2, row = (blk & 3) * 32 + lane;
  const bool finish = mine >= 0 && mine < kPerCta;
  int row_seq = 0, cs = 0;
  const int64_t trow = (int64_t)I * kTT + row;
  if (finish) {
    row_seq = kSampled ? (int)trow : __ldg(p.tokseq + min(trow, p.T - 1));
    cs = __ldg(p.tokseq + min((int64_t)J * kTT + g * 32 + lane, p.T - 1));
  }
  cluster_wait();
  float* const K = h == 0 ? p.K[0] : (h == 1 ? p.K[1] : p.K[2]);
  if (finish && !*abort_flag) {
    // ranks 0 .. np - 1 have sums of P, nq .. C - 1 of Q; the one that has both sent its Q to the last slot
    uint32_t pv[32], qv[32];
    auto add_up = [&](uint32_t (&v)[32], bool second) {
#pragma unroll
      for (int e = 0; e < 32; ++e) v[e] = 0u;
      for (int r = 0; r < kC; ++r) {
        const int a = first_of(r), b = first_of(r + 1);
        if (second ? b <= nkx : a >= nkx) continue;
        const int slot = second && a < nkx ? kC : r;
        const float4* from = reinterpret_cast<const float4*>(sums + (slot * kPerCta + mine) * kBlockBytes) + lane;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const float4 x = from[e * 32];
          v[4 * e] = __float_as_uint(__uint_as_float(v[4 * e]) + x.x);
          v[4 * e + 1] = __float_as_uint(__uint_as_float(v[4 * e + 1]) + x.y);
          v[4 * e + 2] = __float_as_uint(__uint_as_float(v[4 * e + 2]) + x.z);
          v[4 * e + 3] = __float_as_uint(__uint_as_float(v[4 * e + 3]) + x.w);
        }
      }
    };
    add_up(pv, false);
    add_up(qv, true);
    const RowSegments rows = row_segments(row_seq, (long long)(kSampled ? p.n_rows : p.B) * p.B, p.info, !kSampled || trow < (int64_t)p.n_rows);
    int cur = __shfl_sync(0xffffffffu, cs, 0);
    float wseg = (!kSampled && row_seq == cur) ? 2.f : 1.f, run = 0.f;
    gram_group<!kSampled>(pv, qv, cs, g * 32, row, diag, rows, K, p.B, cur, wseg, run);
    flush_rows(K, p.B, rows, cur, run);
  }
  if (!kSampled && p.complete) {
    __threadfence();
    __syncwarp();
    cluster_arrive();
    cluster_wait();
    if (rank == 0 && warp >= 2 && warp < 6) mirror_by_cta<true>(p.K[0], p.B, threadIdx.x - 64, [](int) { return 0.f; }, false);
  }

  if (*abort_flag) __nanosleep(100000);
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem_base, kTmemCols);
}

template <bool kSampled, int kC>
isopo_status launch_split(const CUtensorMap (&maps)[6], const GramSplitParams& p, int n_heads, int id, cudaStream_t st) {
  const auto kernel = &k_bf16_gram_split<kSampled, kC>;
  ISOPO_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, split_smem(kC)));
  {
    LaunchScope scope(id, st);
    launch(kernel, p.units * n_heads * kC, kThreads, split_smem(kC), st, maps[0], maps[1], maps[2], maps[3], maps[4], maps[5], p);
  }
  ISOPO_CUDA_TRY(cudaGetLastError());
  return ISOPO_OK;
}

template <bool kSampled>
isopo_status dispatch(int ctas, const CUtensorMap (&maps)[6], const GramSplitParams& p, int n_heads, int id, cudaStream_t st) {
  switch (ctas) {
    case 2: return launch_split<kSampled, 2>(maps, p, n_heads, id, st);
    case 4: return launch_split<kSampled, 4>(maps, p, n_heads, id, st);
    default: return launch_split<kSampled, 8>(maps, p, n_heads, id, st);
  }
}

template <int kC>
bool placed() {
  const auto kernel = &k_bf16_gram_split<false, kC>;  // its CTAs leave no room for another on their SMs
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kC);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = split_smem(kC);
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = kC;
  attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, split_smem(kC)) == cudaSuccess &&
      cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) == cudaSuccess)
    return n >= 1;
  (void)cudaGetLastError();  // an answer, no failure of the call that asks
  return false;
}

}  // namespace

int placed_cluster(int wanted) {
  if (wanted >= 8 && placed<8>()) return 8;
  if (wanted >= 4 && placed<4>()) return 4;
  return wanted >= 2 && placed<2>() ? 2 : 1;
}

// CTAs per tile: 1 where the kernels of tc_gram.cu and tc_gram_shared.cu are the better.  As many as leave a CTA six stages and
// all clusters resident at one time: clusters of four or eight find fewer than 148 SMs (1000 tokens, 3584 x 8192, 36 tiles: 38.2 us
// one CTA, 28.8 two, 35.7 four).  Whole isopo_layer_gram, one CTA / 2 / 4 / 8: 169 tokens (3 tiles), 3584 x 10752 45.8 / 30.8 / 21.0 /
// 17.5; 480 (10), 896 x 4864 24.0 / 19.6 / 16.8 / 16.2; 800 (28), 2560 x 10240 41.2 / 30.3 / 22.9 / 33.0; 1300 (66), 896 x 896 14.1 /
// 13.4; 300 (6), 512 x 128, ten stages, 13.3 / 14.1 / 14.5 / 14.0; sixteen CTAs gain nothing on eight.
int gram_split_ctas(long long units, int d_in, int d_out, int sms) {
  const int stages = (d_in + kKF - 1) / kKF + (d_out + kKF - 1) / kKF;
  int c = 1;
  while (c < 8 && units * 2 * c <= (c == 1 ? sms : sms * 7 / 8) && stages >= 12 * c) c *= 2;
  return c > 1 ? placed_cluster(c) : 1;
}

isopo_status bf16_gram_split(int ctas, const void* X, int ldx, const void* const* dY, const int* ldy, int64_t T, int d_in, const int* d_out, int n_heads,
                             const int32_t* tokseq, int B, float* const* K, bool complete, int32_t* info, cudaStream_t st) {
  CUtensorMap maps[6];
  isopo_status s = make_map_2d_bf16(&maps[2], X, (uint64_t)T, (uint64_t)d_in, (uint64_t)ldx, 64, kTT);
  GramSplitParams p{};
  for (int h = 0; h < kMaxProj && s == ISOPO_OK; ++h) {
    const int k = h < n_heads ? h : 0;
    s = make_map_2d_bf16(&maps[3 + h], dY[k], (uint64_t)T, (uint64_t)d_out[k], (uint64_t)ldy[k], 64, kTT);
    p.K[h] = K[k];
    p.d_out[h] = d_out[k];
  }
  if (s != ISOPO_OK) return s;
  maps[0] = maps[2];
  maps[1] = maps[3];
  p.tokseq = tokseq; p.T = T; p.B = B; p.nT = (int)((T + kTT - 1) / kTT); p.d_in = d_in; p.info = info;
  p.units = p.nT * (p.nT + 1) / 2;
  p.complete = complete;
  return dispatch<false>(ctas, maps, p, n_heads, kIdGram, st);
}

isopo_status bf16_sampled_split(int ctas, const void* X, const void* dY, int64_t T, int d_in, int d_out, const int32_t* tokseq, int B,
                                const void* A0, int lda, const void* G0, int ldg, int n_samples, float* Mt, int32_t* info, cudaStream_t st) {
  CUtensorMap maps[6];
  isopo_status s;
  if ((s = make_map_2d_bf16(&maps[2], X, (uint64_t)T, (uint64_t)d_in, (uint64_t)d_in, 64, kTT)) != ISOPO_OK) return s;
  if ((s = make_map_2d_bf16(&maps[3], dY, (uint64_t)T, (uint64_t)d_out, (uint64_t)d_out, 64, kTT)) != ISOPO_OK) return s;
  const uint32_t box_rows = sample_box_rows(n_samples);
  if ((s = make_map_2d_bf16(&maps[0], A0, (uint64_t)n_samples, (uint64_t)d_in, (uint64_t)lda, 64, box_rows)) != ISOPO_OK) return s;
  if ((s = make_map_2d_bf16(&maps[1], G0, (uint64_t)n_samples, (uint64_t)d_out, (uint64_t)ldg, 64, box_rows)) != ISOPO_OK) return s;
  maps[4] = maps[5] = maps[3];
  GramSplitParams p{};
  for (int h = 0; h < kMaxProj; ++h) { p.K[h] = Mt; p.d_out[h] = d_out; }
  p.tokseq = tokseq; p.T = T; p.B = B; p.nT = (int)((T + kTT - 1) / kTT); p.d_in = d_in; p.info = info;
  p.n_rows = n_samples;
  p.row_bytes = box_rows * 128;
  p.n_row_tiles = (n_samples + kTT - 1) / kTT;
  p.units = p.nT * p.n_row_tiles;
  return dispatch<true>(ctas, maps, p, 1, kIdSampled, st);
}

}  // namespace isopo
