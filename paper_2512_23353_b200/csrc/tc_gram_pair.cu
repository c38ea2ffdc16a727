// Token-Gram kernel of the Gram route with 2-CTA tensor-core tiles (the 1-CTA kernel of tc_gram.cu states the math: K from the
// elementwise product of P = X X^T and Q = dY dY^T, summed per pair of sequences).
//
// A 128 x 128 tile of one CTA takes 32 KB from L2 into shared memory, and as much from there to the tensor cores, for every
// 64 features, which at the tensor cores' peak is all that shared memory moves.  A pair of CTAs works on 256 x 256 tiles, each
// with its own 128 rows and half of the columns: half the bytes per flop on both ways.
// One tile's P and Q are all of tensor memory, so nothing is double-buffered.  Instead the epilogue takes P into registers (128
// per thread) while the tensor cores form Q; when that is done they go on with the next tile's P, and the epilogue reads Q
// meanwhile.  The wider operand is P's, whose steps have to cover the epilogue.  Projections that share X (tc_gram_shared.cu)
// share P: their Q follow one another through the two halves of tensor memory, P in registers for all of them.
// 896 x 896, 41 tokens per sequence: 10,496 tokens 165 -> 133 us (1.50 PFLOP/s), 40,960 tokens 2.75 -> 2.09 ms (1-CTA tiles with
// the same epilogue -> this); 256 x 128 tiles with two buffers of P and Q: 151 us and 2.36 ms.
//
//   warp 0          TMA producer; both CTAs' copies complete on the barrier in CTA 0
//   warp 1, CTA 0   MMA issuer (one elected thread), tcgen05.mma.cta_group::2 256 x 256 x 16
//   warps 4-11      epilogue (tc_gram_epilogue.cuh): 32 of the CTA's own 128 rows, one of the two 128-column tiles
//
// Every wait is bounded; the teardown is that of tc_seq_grad_pair.cu.
#include <algorithm>
#include <utility>

#include "tc_common.cuh"
#include "tc_gram_epilogue.cuh"

namespace isopo {

namespace {

using namespace tc;

constexpr int kTT = 128;                       // token rows per CTA
constexpr int kKF = 64;                        // features per stage (128 bytes of bf16)
constexpr int kStages = 6;
constexpr int kOperandBytes = kTT * 128;       // 16 KB: the CTA's rows, its half of the columns
constexpr int kStageBytes = 2 * kOperandBytes;
constexpr int kSmemBytes = kStages * kStageBytes + 1024 + 256;
constexpr int kThreads = 384;
// Registers: ten warps would get 168 a thread (three warps on some schedulers), twelve take 64,512 of them and split those
// unevenly: 128 threads of 56 and 256 of 216 are 62,464.  With 168 the epilogue spills: 64 x 416, 40,940 tokens 636 -> 566 us,
// 896 x 896, 10,496 tokens 125.5 -> 123.0.
constexpr int kIssueRegs = 56, kEpilogueRegs = 216;
static_assert(128 * kIssueRegs + 256 * kEpilogueRegs <= kThreads * 168, "the block has no more");
constexpr uint32_t kTmemCols = 512;            // P 256, Q 256
static_assert(kSmemBytes <= 227 * 1024, "shared memory");

constexpr int kMaxHeads = 3;
struct GramPairParams {
  const int32_t* tokseq;
  float* K[kMaxHeads];
  int64_t T;
  int B, nT, nblocks, n_heads, strip;  // nT: 128-token tiles, nblocks: 256-token blocks
  int nk[1 + kMaxHeads];               // 64-feature steps of P and of every Q
  int32_t* info;
};
// no indexing by a run-time value: that would move the parameters to local memory
__device__ __forceinline__ int steps(const GramPairParams& p, int f) {
  return f == 0 ? p.nk[0] : f == 1 ? p.nk[1] : f == 2 ? p.nk[2] : p.nk[3];
}

// kShared: several projections (one by itself has less to keep track of: 256 x 256, 16,000 tokens 99.5 -> 91.6 us).
template <bool kShared>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
k_bf16_gram_pair(const __grid_constant__ CUtensorMap mapP, const __grid_constant__ CUtensorMap mapQ0,
                 const __grid_constant__ CUtensorMap mapQ1, const __grid_constant__ CUtensorMap mapQ2, GramPairParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t smem_base = smem_u32(smem);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kStages * kStageBytes);
  const uint32_t bar0 = smem_u32(bars);
  auto full_bar = [&](int s) { return bar0 + 8u * s; };                          // used in CTA 0
  auto empty_bar = [&](int s) { return bar0 + 8u * (kStages + s); };             // both CTAs
  auto accfull_bar = [&](int b) { return bar0 + 8u * (2 * kStages + b); };       // both CTAs
  auto accempty_bar = [&](int b) { return bar0 + 8u * (2 * kStages + 2 + b); };  // used in CTA 0
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kStages + 4);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const uint32_t peer_abort = map_to_cta(smem_u32(const_cast<int*>(abort_flag)), rank ^ 1u);
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(accfull_bar(b), 1); mbar_init(accempty_bar(b), 16); }
    *abort_flag = 0;
    fence_barrier_init();
  }
  if (warp == 1) tmem_alloc_pair(smem_u32(tmem_slot), kTmemCols);
  pdl_begin();
  tc_fence_before_sync();
  __syncthreads();
  __syncwarp();
  cluster_sync_all();
  tc_fence_after_sync();
  const uint32_t tmem_base = *tmem_slot;

  const unsigned first = blockIdx.x >> 1, step = gridDim.x >> 1;
  const int n_heads = kShared ? p.n_heads : 1;
  // accumulators in turn: P, Q of every projection, P of the next unit, ..: the c-th is half c & 1, its use of it c >> 1

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kIssueRegs));
    if (warp == 0) {
      if (elect_one()) {
        prefetch_tensormap(&mapP);
        prefetch_tensormap(&mapQ0);
        if (n_heads > 1) prefetch_tensormap(&mapQ1);
        if (n_heads > 2) prefetch_tensormap(&mapQ2);
        const uint32_t full_at_leader = map_to_cta(full_bar(0), 0);
        int stage = 0;
        uint32_t phase = 0;
        bool ok = true;
        for (PairWalk u(p.nblocks, p.strip, first); u.more() && ok; u.next(step)) {
          int I, J;
          u.get(I, J);
          const int row = (2 * I + (int)rank) * kTT, col = (2 * J + (int)rank) * kTT;  // tokens past T read as zero
#pragma unroll(kShared ? 1 : 2)
          for (int f = 0; f <= n_heads && ok; ++f) {
            const CUtensorMap* map = f == 0 ? &mapP : f == 1 ? &mapQ0 : f == 2 ? &mapQ1 : &mapQ2;
            const int nk = steps(p, f);
            for (int kb = 0; kb < nk; ++kb) {
              if (!(ok = mbar_wait_pair(empty_bar(stage), phase ^ 1u, abort_flag, peer_abort, p.info, kIdGram))) break;
              const uint32_t dst = smem_base + stage * kStageBytes, fb = full_at_leader + 8u * stage;
              if (rank == 0) mbar_arrive_expect_tx(full_bar(stage), 2 * kStageBytes);
              tma_load_2d_pair(dst, map, kb * kKF, row, fb);
              tma_load_2d_pair(dst + kOperandBytes, map, kb * kKF, col, fb);
              if (++stage == kStages) { stage = 0; phase ^= 1u; }
            }
          }
        }
      }
    } else if (warp == 1) {
      if (rank == 0 && elect_one()) {
        constexpr uint32_t idesc = make_idesc_bf16(2 * kTT, 2 * kTT, false, false);
        int stage = 0;
        uint32_t phase = 0;
        unsigned c = 0;
        bool ok = true;
        for (PairWalk u(p.nblocks, p.strip, first); u.more() && ok; u.next(step)) {
#pragma unroll(kShared ? 1 : 2)
          for (int f = 0; f <= n_heads && ok; ++f, ++c) {
            const unsigned acc = kShared ? c & 1u : (unsigned)f;
            if (!(ok = mbar_wait_pair(accempty_bar(acc), ((c >> 1) & 1u) ^ 1u, abort_flag, peer_abort, p.info, kIdGram))) break;
            tc_fence_after_sync();
            const int nk = steps(p, f);
            for (int kb = 0; kb < nk; ++kb) {
              if (!(ok = mbar_wait_pair(full_bar(stage), phase, abort_flag, peer_abort, p.info, kIdGram))) break;
              tc_fence_after_sync();
              const uint32_t a_addr = smem_base + stage * kStageBytes, b_addr = a_addr + kOperandBytes;
#pragma unroll
              for (int k16 = 0; k16 < kKF / 16; ++k16) {
                const uint64_t a_desc = make_sdesc_sw128(a_addr + k16 * 32, 16, 1024);
                const uint64_t b_desc = make_sdesc_sw128(b_addr + k16 * 32, 16, 1024);
                mma_bf16_pair(tmem_base + acc * 256, a_desc, b_desc, idesc, (kb | k16) != 0);
              }
              mma_commit_pair(empty_bar(stage));
              if (++stage == kStages) { stage = 0; phase ^= 1u; }
            }
            if (ok) mma_commit_pair(accfull_bar(acc));
          }
        }
      }
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kEpilogueRegs));
    const int q = warp & 3, row = q * 32 + lane, half = (warp - 4) / 4;  // 32 rows and one of the two column tiles
    const uint32_t accempty_at_leader = map_to_cta(accempty_bar(0), 0);
    const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)half * kTT;
    unsigned c = 0;
    bool ok = true;
    for (PairWalk u(p.nblocks, p.strip, first); u.more() && ok; u.next(step)) {
      int I, J;
      u.get(I, J);
      I = 2 * I + (int)rank;
      J = 2 * J + half;
      const bool diag = I == J, active = I <= J && J < p.nT;  // else below the diagonal or past the last token
      // sequence of this thread's row token and of the column tokens 32 g + lane (clamped past the end; those rows and columns
      // are zero in P and Q)
      const int row_seq = __ldg(p.tokseq + min((int64_t)I * kTT + row, p.T - 1));
      int cs[kTT / 32];
#pragma unroll
      for (int g = 0; g < kTT / 32; ++g) cs[g] = __ldg(p.tokseq + min((int64_t)J * kTT + g * 32 + lane, p.T - 1));
      const RowSegments rows = row_segments(row_seq, (long long)p.B * p.B, p.info);
      uint32_t pv[kTT / 32][32];
      const unsigned accP = kShared ? c & 1u : 0u;
      if (!mbar_wait_pair(accfull_bar(accP), (c >> 1) & 1u, abort_flag, peer_abort, p.info, kIdGram)) break;
      tc_fence_after_sync();
      if (active) {
#pragma unroll
        for (int g = 0; g < kTT / 32; ++g) tmem_ld32(taddr + accP * 256 + g * 32, pv[g]);
        tmem_ld_wait();
      }
      tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive_remote(accempty_at_leader + 8u * accP);
      ++c;
#pragma unroll 1
      for (int h = 0; h < n_heads; ++h, ++c) {
        const unsigned accQ = kShared ? c & 1u : 1u;
        if (!(ok = mbar_wait_pair(accfull_bar(accQ), (c >> 1) & 1u, abort_flag, peer_abort, p.info, kIdGram))) break;
        tc_fence_after_sync();
        if (active) {
          float* K = h == 0 ? p.K[0] : h == 1 ? p.K[1] : p.K[2];
          int cur = __shfl_sync(0xffffffffu, cs[0], 0);
          float wseg = row_seq == cur ? 2.f : 1.f, run = 0.f;
#pragma unroll
          for (int g = 0; g < kTT / 32; ++g) {
            uint32_t qv[32];
            tmem_ld32(taddr + accQ * 256 + g * 32, qv);
            tmem_ld_wait();
            gram_group<true>(pv[g], qv, cs[g], g * 32, row, diag, rows, K, p.B, cur, wseg, run, kShared && h > 0);
          }
          flush_rows(K, p.B, rows, cur, run);
        }
        tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive_remote(accempty_at_leader + 8u * accQ);
      }
    }
  }

  if (*abort_flag) __nanosleep(100000);
  tc_fence_before_sync();
  __syncthreads();
  __syncwarp();
  cluster_sync_all();
  if (warp == 1) tmem_dealloc_pair(tmem_base, kTmemCols);
}

}  // namespace

// Costs in 64-feature steps of a 1-CTA tile (0.19 us); a wave is a tile per CTA or pair, which its epilogue bounds from below.
// Tiles of 256 x 256 move half the bytes per flop, but take 2.5 us more to set up and drain and give the chip coarser units; a
// pair's wave, twice the tokens per SM, is 1.65 of the other's, 1.45 from about 5000 tokens on.
// Measured (1-CTA / 2-CTA): 896 x 896: 12.4 / 18.1 us at 2048 tokens, 23.6 / 27.3 at 3328, 28.3 / 27.6 at 3840, 33.1 / 35.1 at
// 4352 (5 waves / 3), 39.6 / 36.8 at 5120, 137 / 121 at 10,240; 896 x 4864: 54.3 / 63.2 at 3328, 69.1 / 63.3 at 3840, 85.6 /
// 89.2 at 4352, 429 / 395 at 10,240; 448 x 448: 19.0 / 19.1 at 3840, 31.4 / 33.2 at 6144, 142 / 119 at 14,336; 256 x 256: 35.6 /
// 36.5 at 8192, 89.4 / 80.7 at 14,336; 128 x 64: 58 / 65 at 14,336; 64 x 416: 792 / 641 at 40,940.
bool bf16_gram_pair_pays(int64_t T, int d_in, const int* d_out, int n_heads, int sms) {
  long long nk = (d_in + kKF - 1) / kKF;
  for (int h = 0; h < n_heads; ++h) nk += (d_out[h] + kKF - 1) / kKF;
  const long long nT = (T + kTT - 1) / kTT, nb = (nT + 1) / 2, pairs = sms / 2;
  const long long waves = (nT * (nT + 1) / 2 + sms - 1) / sms, pair_waves = (nb * (nb + 1) / 2 + pairs - 1) / pairs;
  return pair_waves * std::max((pair_waves >= 5 ? 1.45 : 1.65) * nk, 14.0 * n_heads) + 12 < waves * std::max((double)nk, 6.5 * n_heads);
}

isopo_status bf16_gram_pair(const void* X, int ldx, const void* const* dY, const int* ldy, int64_t T, int d_in, const int* d_out, int n_heads,
                            const int32_t* tokseq, int B, float* const* K, int32_t* info, cudaStream_t st) {
  if (n_heads < 1 || n_heads > kMaxHeads) return ISOPO_ERR_INVALID_ARG;
  // P o Q = Q o P: of one projection the wider operand goes first
  const void* operand[1 + kMaxHeads] = {X, dY[0]};
  int d[1 + kMaxHeads] = {d_in, d_out[0]}, ld[1 + kMaxHeads] = {ldx, ldy[0]}, d_sum = 0;
  if (n_heads == 1 && d[1] > d[0]) {
    std::swap(operand[0], operand[1]);
    std::swap(d[0], d[1]);
    std::swap(ld[0], ld[1]);
  }
  GramPairParams p{};
  for (int h = 1; h < n_heads; ++h) { operand[1 + h] = dY[h]; d[1 + h] = d_out[h]; ld[1 + h] = ldy[h]; }
  CUtensorMap map[1 + kMaxHeads];
  for (int f = 0; f <= kMaxHeads; ++f) {
    const int ff = std::min(f, n_heads);  // unused slots repeat the last projection's map
    isopo_status s = make_map_2d_bf16(&map[f], operand[ff], (uint64_t)T, (uint64_t)d[ff], (uint64_t)ld[ff], 64, kTT);
    if (s != ISOPO_OK) return s;
    if (f > n_heads) continue;
    p.nk[f] = (d[f] + kKF - 1) / kKF;
    d_sum += d[f];
    if (f > 0) p.K[f - 1] = K[f - 1];
  }
  int dev = 0, sms = 0;
  ISOPO_CUDA_TRY(cudaGetDevice(&dev));
  ISOPO_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const auto kernel = n_heads > 1 ? &k_bf16_gram_pair<true> : &k_bf16_gram_pair<false>;
  ISOPO_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes));
  p.tokseq = tokseq; p.T = T; p.B = B; p.n_heads = n_heads; p.info = info;
  p.nT = (int)((T + kTT - 1) / kTT);
  p.nblocks = (p.nT + 1) / 2;
  const long long units = (long long)p.nblocks * (p.nblocks + 1) / 2;
  const int pairs = (int)std::min<long long>(units, sms / 2);
  p.strip = gram_strip_width(2.0 * 2 * kTT * d_sum, pairs);
  {
    LaunchScope scope(kIdGram, st);
    launch(kernel, 2 * pairs, kThreads, kSmemBytes, st, map[0], map[1], map[2], map[3], p);
  }
  ISOPO_CUDA_TRY(cudaGetLastError());
  for (int h = 0; h < n_heads; ++h) {
    isopo_status s = mirror_upper(K[h], B, st);
    if (s != ISOPO_OK) return s;
  }
  return ISOPO_OK;
}

}  // namespace isopo
