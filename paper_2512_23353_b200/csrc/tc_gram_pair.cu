// Token-Gram kernel of the Gram route with 2-CTA tensor-core tiles (the 1-CTA kernel of tc_gram.cu states the math: K from the
// elementwise product of P = X X^T and Q = dY dY^T, summed per pair of sequences).
//
// A 128 x 128 tile of one CTA takes 32 KB from L2 into shared memory, and as much from there to the tensor cores, for every
// 64 features, which at the tensor cores' peak is all that shared memory moves.  A pair of CTAs works on 256 x 256 tiles, each
// with its own 128 rows and half of the columns: half the bytes per flop on both ways.
// One tile's P and Q are all of tensor memory, so nothing is double-buffered.  Instead the epilogue takes P into registers (128
// per thread) while the tensor cores form Q; when that is done they go on with the next tile's P, and the epilogue reads Q
// meanwhile.  The wider operand is P's, whose steps have to cover the epilogue.
// 896 x 896, 41 tokens per sequence: 10,496 tokens 165 -> 133 us (1.50 PFLOP/s), 40,960 tokens 2.75 -> 2.09 ms (1-CTA tiles with
// the same epilogue -> this); 256 x 128 tiles with two buffers of P and Q: 151 us and 2.36 ms.
//
//   warp 0          TMA producer; both CTAs' copies complete on the barrier in CTA 0
//   warp 1, CTA 0   MMA issuer (one elected thread), tcgen05.mma.cta_group::2 256 x 256 x 16
//   warps 2-9       epilogue (tc_gram_epilogue.cuh): 32 of the CTA's own 128 rows, one of the two 128-column tiles
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
constexpr int kThreads = 320;
constexpr uint32_t kTmemCols = 512;            // P 256, Q 256
static_assert(kSmemBytes <= 227 * 1024, "shared memory");

struct GramPairParams {
  const int32_t* tokseq;
  float* K;
  int64_t T;
  int B, nT, nblocks, d_p, d_q, strip;  // nT: 128-token tiles, nblocks: 256-token blocks
  int32_t* info;
};

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
k_bf16_gram_pair(const __grid_constant__ CUtensorMap mapP, const __grid_constant__ CUtensorMap mapQ, GramPairParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t smem_base = smem_u32(smem);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kStages * kStageBytes);
  const uint32_t bar0 = smem_u32(bars);
  auto full_bar = [&](int s) { return bar0 + 8u * s; };                          // used in CTA 0
  auto empty_bar = [&](int s) { return bar0 + 8u * (kStages + s); };             // both CTAs
  auto accfull_bar = [&](int b) { return bar0 + 8u * (2 * kStages + b); };       // P, Q; both CTAs
  auto accempty_bar = [&](int b) { return bar0 + 8u * (2 * kStages + 2 + b); };  // P, Q; used in CTA 0
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
  const int nkp = (p.d_p + kKF - 1) / kKF, nkq = (p.d_q + kKF - 1) / kKF;

  if (warp == 0) {
    if (elect_one()) {
      prefetch_tensormap(&mapP);
      prefetch_tensormap(&mapQ);
      const uint32_t full_at_leader = map_to_cta(full_bar(0), 0);
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      for (PairWalk u(p.nblocks, p.strip, first); u.more() && ok; u.next(step)) {
        int I, J;
        u.get(I, J);
        const int row = (2 * I + (int)rank) * kTT, col = (2 * J + (int)rank) * kTT;  // tokens past T read as zero
        for (int kb = 0; kb < nkp + nkq; ++kb) {
          if (!(ok = mbar_wait_pair(empty_bar(stage), phase ^ 1u, abort_flag, peer_abort, p.info, kIdGram))) break;
          const CUtensorMap* map = kb < nkp ? &mapP : &mapQ;
          const int x = (kb < nkp ? kb : kb - nkp) * kKF;
          const uint32_t dst = smem_base + stage * kStageBytes, fb = full_at_leader + 8u * stage;
          if (rank == 0) mbar_arrive_expect_tx(full_bar(stage), 2 * kStageBytes);
          tma_load_2d_pair(dst, map, x, row, fb);
          tma_load_2d_pair(dst + kOperandBytes, map, x, col, fb);
          if (++stage == kStages) { stage = 0; phase ^= 1u; }
        }
      }
    }
  } else if (warp == 1) {
    if (rank == 0 && elect_one()) {
      constexpr uint32_t idesc = make_idesc_bf16(2 * kTT, 2 * kTT, false, false);
      int stage = 0;
      uint32_t phase = 0, unit_phase = 0;
      bool ok = true;
      for (PairWalk u(p.nblocks, p.strip, first); u.more() && ok; u.next(step)) {
        for (int kb = 0; kb < nkp + nkq; ++kb) {
          const int acc = kb >= nkp, kk = acc ? kb - nkp : kb;
          if (kk == 0) {
            if (!(ok = mbar_wait_pair(accempty_bar(acc), unit_phase ^ 1u, abort_flag, peer_abort, p.info, kIdGram))) break;
            tc_fence_after_sync();
          }
          if (!(ok = mbar_wait_pair(full_bar(stage), phase, abort_flag, peer_abort, p.info, kIdGram))) break;
          tc_fence_after_sync();
          const uint32_t a_addr = smem_base + stage * kStageBytes, b_addr = a_addr + kOperandBytes;
#pragma unroll
          for (int k16 = 0; k16 < kKF / 16; ++k16) {
            const uint64_t a_desc = make_sdesc_sw128(a_addr + k16 * 32, 16, 1024);
            const uint64_t b_desc = make_sdesc_sw128(b_addr + k16 * 32, 16, 1024);
            mma_bf16_pair(tmem_base + (uint32_t)acc * 256, a_desc, b_desc, idesc, (kk | k16) != 0);
          }
          mma_commit_pair(empty_bar(stage));
          if (kk == (acc ? nkq : nkp) - 1) mma_commit_pair(accfull_bar(acc));
          if (++stage == kStages) { stage = 0; phase ^= 1u; }
        }
        unit_phase ^= 1u;
      }
    }
  } else {
    const int q = warp & 3, row = q * 32 + lane, half = (warp - 2) / 4;  // 32 rows and one of the two column tiles
    const uint32_t accempty_at_leader = map_to_cta(accempty_bar(0), 0);
    const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)half * kTT;
    uint32_t phase = 0;
    for (PairWalk u(p.nblocks, p.strip, first); u.more(); u.next(step), phase ^= 1u) {
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
      if (!mbar_wait_pair(accfull_bar(0), phase, abort_flag, peer_abort, p.info, kIdGram)) break;
      tc_fence_after_sync();
      if (active) {
#pragma unroll
        for (int g = 0; g < kTT / 32; ++g) tmem_ld32(taddr + g * 32, pv[g]);
        tmem_ld_wait();
      }
      tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive_remote(accempty_at_leader);
      if (!mbar_wait_pair(accfull_bar(1), phase, abort_flag, peer_abort, p.info, kIdGram)) break;
      tc_fence_after_sync();
      if (active) {
        int cur = __shfl_sync(0xffffffffu, cs[0], 0);
        float wseg = row_seq == cur ? 2.f : 1.f, run = 0.f;
#pragma unroll
        for (int g = 0; g < kTT / 32; ++g) {
          uint32_t qv[32];
          tmem_ld32(taddr + 256 + g * 32, qv);
          tmem_ld_wait();
          gram_group<true>(pv[g], qv, cs[g], g * 32, row, diag, rows, p.K, p.B, cur, wseg, run);
        }
        flush_rows(p.K, p.B, rows, cur, run);
      }
      tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive_remote(accempty_at_leader + 8u);
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

isopo_status bf16_gram_pair(const void* X, const void* dY, int64_t T, int d_in, int d_out, const int32_t* tokseq, int B,
                            float* K, int32_t* info, cudaStream_t st) {
  if (d_out > d_in) {  // P o Q = Q o P
    std::swap(X, dY);
    std::swap(d_in, d_out);
  }
  CUtensorMap mapP, mapQ;
  isopo_status s = make_map_2d_bf16(&mapP, X, (uint64_t)T, (uint64_t)d_in, (uint64_t)d_in, 64, kTT);
  if (s != ISOPO_OK) return s;
  s = make_map_2d_bf16(&mapQ, dY, (uint64_t)T, (uint64_t)d_out, (uint64_t)d_out, 64, kTT);
  if (s != ISOPO_OK) return s;
  int dev = 0, sms = 0;
  ISOPO_CUDA_TRY(cudaGetDevice(&dev));
  ISOPO_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  ISOPO_CUDA_TRY(cudaFuncSetAttribute(k_bf16_gram_pair, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes));
  GramPairParams p{tokseq, K, T, B, (int)((T + kTT - 1) / kTT), (int)((T + 2 * kTT - 1) / (2 * kTT)), d_in, d_out, 0, info};
  const long long units = (long long)p.nblocks * (p.nblocks + 1) / 2;
  const int pairs = (int)std::min<long long>(units, sms / 2);
  p.strip = gram_strip_width(2.0 * 2 * kTT * (d_in + d_out), pairs);
  {
    LaunchScope scope(kIdGram, st);
    launch(k_bf16_gram_pair, 2 * pairs, kThreads, kSmemBytes, st, mapP, mapQ, p);
  }
  ISOPO_CUDA_TRY(cudaGetLastError());
  return mirror_upper(K, B, st);
}

}  // namespace isopo
