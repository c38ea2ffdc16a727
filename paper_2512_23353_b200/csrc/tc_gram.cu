// Gram route to the layer NTK on the tensor cores.
//
// Every token gradient is the rank-one matrix dY_t x_t^T (Eq. one / Eq. two), hence
//   K_ij = sum_{t in i, s in j} (dY_t . dY_s)(x_t . x_s) = [ S ((dY dY^T) o (X X^T)) S^T ]_ij
// with S the B x T sequence indicator.  For a pair of 128-token tiles (I <= J) this kernel forms
// P = X_I X_J^T (contraction over d_in) and Q = dY_I dY_J^T (contraction over d_out) as two
// 128 x 128 float32 accumulators in tensor memory, and its epilogue multiplies them elementwise and
// adds the products into K by (sequence of row token, sequence of column token).  Neither T x T
// matrix ever leaves the SM.
//
// Only token pairs t <= s are visited.  A pair t < s inside one sequence stands for (t,s) and
// (s,t) and counts twice; a pair across sequences i < j lands in K_ij once (K_ji is mirrored at the
// end); t = s counts once.
//
//   warp 0      TMA producer: [128 tokens] x [64 features] boxes of X then of dY, 6-stage ring
//   warp 1      MMA issuer: tcgen05.mma 128 x 128 x 16, K-major operands
//   warps 2-9   epilogue: tcgen05.ld of P and Q, product, segmented sums, float atomics into K
//               (a warp takes 32 rows and half of the columns)

#include "tc_common.cuh"
#include "tc_gram_epilogue.cuh"

namespace isopo {

namespace {

using namespace tc;

constexpr int kTT = 128;                       // tokens per tile
constexpr int kKF = 64;                        // features per stage (128 bytes of bf16)
constexpr int kStages = 6;
constexpr int kOperandBytes = kTT * 128;       // 16 KB
constexpr int kStageBytes = 2 * kOperandBytes;
constexpr int kSmemBytes = kStages * kStageBytes + 1024 + 256;
// Copy warp, MMA warp, eight epilogue warps.  With four and a walk over the units from the beginning for each, the epilogue
// bound every layer of narrow operands or short sequences (128 x 64, 64 tokens each: 15.4 -> 11.9 us at 3840 tokens, 376 -> 207
// at 28,800) and took 1 us longer behind the last MMA of any (896 x 896, 640 tokens: 11.1 -> 10.3).
constexpr int kThreads = 320;
constexpr uint32_t kTmemCols = 512;            // 2 buffers x (P 128 + Q 128) columns

struct GramParams {
  const int32_t* tokseq;
  float* K;       // Gram: K [B, B];  sampled: M^T [samples, B]
  int64_t T;
  int B, nT, d_in, d_out;
  int32_t* info;
  int n_rows, n_row_tiles;  // sampled: sample rows and their 128-row tiles
  int strip;                // Gram: tile columns per strip of the pair order
  uint32_t row_bytes;       // sampled: of a stage's row operand (fewer than 128 samples: no more rows than there are)
};

// The work units of a CTA: (row tile I, column tile J).  Gram: pairs I <= J of token tiles.
// Sampled: every (sample tile, token tile).
template <bool kSampled> struct Units : PairWalk {
  __device__ __forceinline__ Units(const GramParams& p) : PairWalk(p.nT, p.strip, blockIdx.x) {}
  __device__ __forceinline__ void next() { PairWalk::next(gridDim.x); }
};
template <> struct Units<true> {
  int rows, cols, I, J, step_i, step_j;
  __device__ __forceinline__ Units(const GramParams& p)
      : rows(p.n_row_tiles), cols(p.nT), I(blockIdx.x % rows), J(blockIdx.x / rows), step_i(gridDim.x % rows), step_j(gridDim.x / rows) {}
  __device__ __forceinline__ bool more() const { return J < cols; }
  __device__ __forceinline__ void next() {
    I += step_i;
    J += step_j;
    if (I >= rows) { I -= rows; ++J; }
  }
  __device__ __forceinline__ void get(int& i, int& j) const { i = I; j = J; }
};

// kSampled = false: the Gram route, rows and columns are both token tiles (mapRX = mapX, mapRY = mapY).
// kSampled = true: the token-sampled Fisher estimator of Algorithm 1: the rows are the sampled token
// rows a0 = X[samples] (mapRX) and g0 = dY[samples] (mapRY), the columns all tokens, and
//   M^T[j, i] = sum_{t in sequence i} (g0_j . dY_t)(a0_j . x_t) = g0_j . G_i a0_j      (Eq. one)
// comes out of the same product-and-segment-sum epilogue without any symmetry weights.
// kComplete (one CTA): fills K's other triangle as well.
template <bool kSampled, bool kComplete>
__global__ void __launch_bounds__(kThreads, 1)
k_bf16_gram(const __grid_constant__ CUtensorMap mapRX, const __grid_constant__ CUtensorMap mapRY,
            const __grid_constant__ CUtensorMap mapX, const __grid_constant__ CUtensorMap mapY, GramParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t smem_base = smem_u32(smem);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kStages * kStageBytes);
  const uint32_t bar0 = smem_u32(bars);
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (kStages + s); };
  auto accfull_bar = [&](int b) { return bar0 + 8u * (2 * kStages + b); };
  auto accempty_bar = [&](int b) { return bar0 + 8u * (2 * kStages + 2 + b); };
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kStages + 4);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(accfull_bar(b), 1); mbar_init(accempty_bar(b), 8); }
    *abort_flag = 0;
    fence_barrier_init();
  }
  if (warp == 1) tmem_alloc(smem_u32(tmem_slot), kTmemCols);
  pdl_begin();
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem_base = *tmem_slot;

  const int nkx = (p.d_in + kKF - 1) / kKF, nky = (p.d_out + kKF - 1) / kKF;

  if (warp == 0) {
    if (elect_one()) {
      prefetch_tensormap(&mapX);
      prefetch_tensormap(&mapY);
      if (kSampled) {
        prefetch_tensormap(&mapRX);
        prefetch_tensormap(&mapRY);
      }
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      for (Units<kSampled> u(p); u.more() && ok; u.next()) {
        int I, J;
        u.get(I, J);
        const bool diag = !kSampled && I == J;
        for (int kb = 0; kb < nkx + nky; ++kb) {
          if (!(ok = mbar_wait(empty_bar(stage), phase ^ 1u, abort_flag, p.info, kIdGram))) break;
          const CUtensorMap* rmap = kb < nkx ? &mapRX : &mapRY;
          const CUtensorMap* cmap = kb < nkx ? &mapX : &mapY;
          const int x = (kb < nkx ? kb : kb - nkx) * kKF;
          const uint32_t dst = smem_base + stage * kStageBytes;
          mbar_arrive_expect_tx(full_bar(stage), kSampled ? p.row_bytes + kOperandBytes : diag ? kOperandBytes : kStageBytes);
          tma_load_2d(dst, rmap, x, I * kTT, full_bar(stage));
          if (!diag) tma_load_2d(dst + kOperandBytes, cmap, x, J * kTT, full_bar(stage));
          if (++stage == kStages) { stage = 0; phase ^= 1u; }
        }
      }
    }
  } else if (warp == 1) {
    if (elect_one()) {  // elected, not "lane 0": lets the compiler keep the MMA operands in uniform registers
      constexpr uint32_t idesc = make_idesc_bf16(kTT, kTT, false, false);
      int stage = 0, acc = 0;
      uint32_t phase = 0, acc_phase = 0;
      bool ok = true;
      for (Units<kSampled> u(p); u.more() && ok; u.next()) {
        int I, J;
        u.get(I, J);
        const bool diag = !kSampled && I == J;
        if (!(ok = mbar_wait(accempty_bar(acc), acc_phase ^ 1u, abort_flag, p.info, kIdGram))) break;
        tc_fence_after_sync();
        for (int kb = 0; kb < nkx + nky; ++kb) {
          if (!(ok = mbar_wait(full_bar(stage), phase, abort_flag, p.info, kIdGram))) break;
          tc_fence_after_sync();
          const uint32_t a_addr = smem_base + stage * kStageBytes;
          const uint32_t b_addr = diag ? a_addr : a_addr + kOperandBytes;
          const bool second = kb >= nkx;  // accumulating Q
          const uint32_t d_tmem = tmem_base + (uint32_t)acc * 256 + (second ? 128u : 0u);
          const int kk = second ? kb - nkx : kb;
#pragma unroll
          for (int k16 = 0; k16 < kKF / 16; ++k16) {
            const uint64_t a_desc = make_sdesc_sw128(a_addr + k16 * 32, 16, 1024);
            const uint64_t b_desc = make_sdesc_sw128(b_addr + k16 * 32, 16, 1024);
            mma_bf16(d_tmem, a_desc, b_desc, idesc, (kk | k16) != 0);
          }
          mma_commit(empty_bar(stage));
          if (++stage == kStages) { stage = 0; phase ^= 1u; }
        }
        if (!ok) break;
        mma_commit(accfull_bar(acc));
        if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
      }
    }
  } else {
    // a warp takes 32 rows (the TMEM lanes it can read) and half of the columns
    const int q = warp & 3, row = q * 32 + lane, g0 = (warp - 2) / 4 * (kTT / 64);
    int acc = 0;
    uint32_t acc_phase = 0;
    for (Units<kSampled> u(p); u.more(); u.next()) {
      int I, J;
      u.get(I, J);
      const bool diag = !kSampled && I == J;
      // sequence of this thread's row token and of every column token (clamped past the end; those
      // rows and columns are zero in P and Q)
      // (sampled: the "row sequence" is the sample index, its results go to row `row_seq` of M^T;
      // rows past the last sample are zero in P and Q, and they are barred from writing outright: a
      // non-finite input would turn their zeros into NaN, and row `trow` of M^T does not exist)
      const int64_t trow = (int64_t)I * kTT + row;
      const int row_seq = kSampled ? (int)trow : __ldg(p.tokseq + min(trow, p.T - 1));
      auto col_seq = [&](int g) { return __ldg(p.tokseq + min((int64_t)J * kTT + g * 32 + lane, p.T - 1)); };
      int cs = col_seq(g0);  // sequence of column token 32 g + lane
      if (!mbar_wait(accfull_bar(acc), acc_phase, abort_flag, p.info, kIdGram)) break;
      tc_fence_after_sync();
      const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)acc * 256;
      const RowSegments rows = row_segments(row_seq, (long long)(kSampled ? p.n_rows : p.B) * p.B, p.info, !kSampled || trow < (int64_t)p.n_rows);
      int cur = __shfl_sync(0xffffffffu, cs, 0);
      float wseg = (!kSampled && row_seq == cur) ? 2.f : 1.f, run = 0.f;
#pragma unroll 1
      for (int g = g0; g < g0 + kTT / 64; ++g) {
        const int cs_next = g + 1 < g0 + kTT / 64 ? col_seq(g + 1) : 0;
        uint32_t pv[32], qv[32];
        tmem_ld32(taddr + g * 32, pv);
        tmem_ld32(taddr + 128 + g * 32, qv);
        tmem_ld_wait();
        gram_group<!kSampled>(pv, qv, cs, g * 32, row, diag, rows, p.K, p.B, cur, wseg, run);
        cs = cs_next;
      }
      flush_rows(p.K, p.B, rows, cur, run);
      tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(accempty_bar(acc));
      if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
    }
    if (kComplete) {
      __threadfence();
      asm volatile("bar.sync 1, 256;" ::: "memory");  // the epilogue warps
      if (g0 == 0) mirror_by_cta<true>(p.K, p.B, row, [](int) { return 0.f; }, false);
    }
  }

  if (*abort_flag) __nanosleep(100000);
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem_base, kTmemCols);
}


}  // namespace

isopo_status bf16_gram(const void* X, int ldx, const void* dY, int ldy, int64_t T, int d_in, int d_out, const int32_t* tokseq, int B,
                       float* K, int32_t* info, cudaStream_t st) {
  int dev = 0, sms = 0;
  ISOPO_CUDA_TRY(cudaGetDevice(&dev));
  ISOPO_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  GramParams p{tokseq, K, T, B, (int)((T + kTT - 1) / kTT), d_in, d_out, info, 0, 0, 0};
  const long long units = (long long)p.nT * (p.nT + 1) / 2;
  const int grid = (int)std::min<long long>(units, sms), ctas = gram_split_ctas(units, d_in, d_out, sms);
  if (ctas > 1) {
    const isopo_status r = bf16_gram_split(ctas, X, ldx, &dY, &ldy, T, d_in, &d_out, 1, tokseq, B, &K, units == 1 && B <= 32, info, st);
    return r != ISOPO_OK || (units == 1 && B <= 32) ? r : mirror_upper(K, B, st);
  }
  CUtensorMap mapX, mapY;
  isopo_status s = make_map_2d_bf16(&mapX, X, (uint64_t)T, (uint64_t)d_in, (uint64_t)ldx, 64, kTT);
  if (s != ISOPO_OK) return s;
  s = make_map_2d_bf16(&mapY, dY, (uint64_t)T, (uint64_t)d_out, (uint64_t)ldy, 64, kTT);
  if (s != ISOPO_OK) return s;
  if (bf16_gram_pair_pays(T, d_in, &d_out, 1, sms)) return bf16_gram_pair(X, ldx, &dY, &ldy, T, d_in, &d_out, 1, tokseq, B, &K, info, st);
  // One tile of tokens: its CTA completes K, a launch less for the host, which bounds so small a layer (26 tokens, 640 x 280:
  // 29.1 -> 26.4 us with the scaling pass's).  The last of several CTAs would be 0.7 (15 CTAs) to 1.3 us (136) slower than a
  // kernel that is already set up when this one ends, and above 32 sequences so is one CTA.
  const bool complete = grid == 1 && B <= 32;
  const auto kernel = complete ? &k_bf16_gram<false, true> : &k_bf16_gram<false, false>;
  ISOPO_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes));
  p.strip = gram_strip_width(2.0 * kTT * (d_in + d_out), grid);
  {
    LaunchScope scope(kIdGram, st);
    launch(kernel, grid, kThreads, kSmemBytes, st, mapX, mapY, mapX, mapY, p);
  }
  ISOPO_CUDA_TRY(cudaGetLastError());
  return complete ? ISOPO_OK : mirror_upper(K, B, st);
}

isopo_status bf16_sampled(const void* X, const void* dY, int64_t T, int d_in, int d_out, const int32_t* tokseq, int B,
                          const void* A0, int lda, const void* G0, int ldg, int n_samples, float* Mt, int32_t* info, cudaStream_t st) {
  int dev = 0, sms = 0;
  ISOPO_CUDA_TRY(cudaGetDevice(&dev));
  ISOPO_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int ctas = gram_split_ctas((T + kTT - 1) / kTT * ((n_samples + kTT - 1) / kTT), d_in, d_out, sms);
  if (ctas > 1) return bf16_sampled_split(ctas, X, dY, T, d_in, d_out, tokseq, B, A0, lda, G0, ldg, n_samples, Mt, info, st);
  CUtensorMap mapX, mapY, mapRX, mapRY;
  isopo_status s = make_map_2d_bf16(&mapX, X, (uint64_t)T, (uint64_t)d_in, (uint64_t)d_in, 64, kTT);
  if (s != ISOPO_OK) return s;
  if ((s = make_map_2d_bf16(&mapY, dY, (uint64_t)T, (uint64_t)d_out, (uint64_t)d_out, 64, kTT)) != ISOPO_OK) return s;
  const uint32_t box_rows = sample_box_rows(n_samples);
  if ((s = make_map_2d_bf16(&mapRX, A0, (uint64_t)n_samples, (uint64_t)d_in, (uint64_t)lda, 64, box_rows)) != ISOPO_OK) return s;
  if ((s = make_map_2d_bf16(&mapRY, G0, (uint64_t)n_samples, (uint64_t)d_out, (uint64_t)ldg, 64, box_rows)) != ISOPO_OK) return s;
  ISOPO_CUDA_TRY(cudaFuncSetAttribute(k_bf16_gram<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes));
  GramParams p{tokseq, Mt, T, B, (int)((T + kTT - 1) / kTT), d_in, d_out, info, n_samples, (n_samples + kTT - 1) / kTT, 0};
  p.row_bytes = box_rows * 128;
  const long long units = (long long)p.n_row_tiles * p.nT;
  const int grid = (int)std::min<long long>(units, sms);
  {
    LaunchScope scope(kIdSampled, st);
    launch(k_bf16_gram<true, false>, grid, kThreads, kSmemBytes, st, mapRX, mapRY, mapX, mapY, p);
  }
  ISOPO_CUDA_TRY(cudaGetLastError());
  return ISOPO_OK;
}

}  // namespace isopo
