// Token-Gram kernel of the Gram route with 2-CTA tensor-core tiles (the 1-CTA kernel of tc_gram.cu states the math: K from the
// elementwise product of P = X X^T and Q = dY dY^T, summed per pair of sequences).
//
// The 1-CTA kernel loads two 16 KB operand tiles for every 128 x 128 x 64 step, 128 bytes per SM and cycle of the tensor
// cores at their peak, and is bound by that.  A pair of CTAs works on 256 x 128 tiles: each loads its own 128 rows and half of
// the 128 columns, 24 KB per step.  P and Q are 128 columns of tensor memory each in both CTAs, so two units still fit and a
// unit's epilogue is overlapped with the next one's MMAs (256 x 256 tiles would need all of it for one unit).
//
// Units: 256 x 256 blocks I <= J of token pairs in strip order, each cut into its two column halves.
//
//   warp 0          TMA producer; both CTAs' copies complete on the barrier in CTA 0
//   warp 1, CTA 0   MMA issuer (one elected thread), tcgen05.mma.cta_group::2 256 x 128 x 16
//   warps 2-9       epilogue (tc_gram_epilogue.cuh), each CTA for its own 128 rows
//
// Every wait is bounded; the teardown is that of tc_seq_grad_pair.cu.
#include <algorithm>

#include "tc_common.cuh"
#include "tc_gram_epilogue.cuh"

namespace isopo {

namespace {

using namespace tc;

constexpr int kTT = 128;                         // tokens per tile and CTA
constexpr int kKF = 64;                          // features per stage (128 bytes of bf16)
constexpr int kStages = 8;
constexpr int kRowBytes = kTT * 128;             // a CTA's rows: 16 KB
constexpr int kColBytes = kTT / 2 * 128;         // its half of the columns: 8 KB
constexpr int kStageBytes = kRowBytes + kColBytes;
constexpr int kSmemBytes = kStages * kStageBytes + 1024 + 256;
constexpr int kEpiWarps = 8;
constexpr int kThreads = 64 + 32 * kEpiWarps;
constexpr int kGroups = kTT / 32 / (kEpiWarps / 4);  // 32-column groups of an epilogue warp
constexpr uint32_t kTmemCols = 512;              // 2 buffers x (P 128 + Q 128) columns
static_assert(kSmemBytes <= 227 * 1024, "shared memory");

struct GramPairParams {
  const int32_t* tokseq;
  float* K;
  int64_t T;
  int B, nT, nblocks, d_in, d_out, strip;  // nblocks: 256-token blocks
  int32_t* info;
};

// The units of a pair of CTAs: (block row I, tile column J), two neighbouring pairs take the two halves of a block.  A half
// whose columns lie past the last token is no unit.
struct Units {
  PairWalk blocks;
  unsigned unit, step;
  int nT;
  __device__ __forceinline__ Units(const GramPairParams& p)
      : blocks(p.nblocks, p.strip, blockIdx.x >> 2), unit(blockIdx.x >> 1), step(gridDim.x >> 1), nT(p.nT) {
    int I, J;
    if (more() && !get(I, J)) next();
  }
  __device__ __forceinline__ bool more() const { return blocks.more(); }
  __device__ __forceinline__ bool get(int& I, int& J) const {
    blocks.get(I, J);
    J = 2 * J + (int)(unit & 1u);
    return J < nT;
  }
  __device__ __forceinline__ void next() {
    int I, J;
    do {
      const unsigned to = unit + step;
      blocks.next((to >> 1) - (unit >> 1));
      unit = to;
    } while (more() && !get(I, J));
  }
};

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
k_bf16_gram_pair(const __grid_constant__ CUtensorMap mapRX, const __grid_constant__ CUtensorMap mapRY,
                 const __grid_constant__ CUtensorMap mapCX, const __grid_constant__ CUtensorMap mapCY, GramPairParams p) {
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
    for (int b = 0; b < 2; ++b) { mbar_init(accfull_bar(b), 1); mbar_init(accempty_bar(b), 2 * kEpiWarps); }
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

  const int nkx = (p.d_in + kKF - 1) / kKF, nky = (p.d_out + kKF - 1) / kKF;

  if (warp == 0) {
    if (elect_one()) {
      prefetch_tensormap(&mapRX);
      prefetch_tensormap(&mapRY);
      prefetch_tensormap(&mapCX);
      prefetch_tensormap(&mapCY);
      const uint32_t full_at_leader = map_to_cta(full_bar(0), 0);
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      for (Units u(p); u.more() && ok; u.next()) {
        int I, J;
        u.get(I, J);
        const int row = (2 * I + (int)rank) * kTT, col = J * kTT + (int)rank * (kTT / 2);  // tokens past T read as zero
        for (int kb = 0; kb < nkx + nky; ++kb) {
          if (!(ok = mbar_wait_pair(empty_bar(stage), phase ^ 1u, abort_flag, peer_abort, p.info, kIdGram))) break;
          const bool first = kb < nkx;
          const int x = (first ? kb : kb - nkx) * kKF;
          const uint32_t dst = smem_base + stage * kStageBytes, fb = full_at_leader + 8u * stage;
          if (rank == 0) mbar_arrive_expect_tx(full_bar(stage), 2 * kStageBytes);
          tma_load_2d_pair(dst, first ? &mapRX : &mapRY, x, row, fb);
          tma_load_2d_pair(dst + kRowBytes, first ? &mapCX : &mapCY, x, col, fb);
          if (++stage == kStages) { stage = 0; phase ^= 1u; }
        }
      }
    }
  } else if (warp == 1) {
    if (rank == 0 && elect_one()) {
      constexpr uint32_t idesc = make_idesc_bf16(2 * kTT, kTT, false, false);
      int stage = 0, acc = 0;
      uint32_t phase = 0, acc_phase = 0;
      bool ok = true;
      for (Units u(p); u.more() && ok; u.next()) {
        int I, J;
        u.get(I, J);
        if (!(ok = mbar_wait_pair(accempty_bar(acc), acc_phase ^ 1u, abort_flag, peer_abort, p.info, kIdGram))) break;
        tc_fence_after_sync();
        for (int kb = 0; kb < nkx + nky; ++kb) {
          if (!(ok = mbar_wait_pair(full_bar(stage), phase, abort_flag, peer_abort, p.info, kIdGram))) break;
          tc_fence_after_sync();
          const uint32_t a_addr = smem_base + stage * kStageBytes, b_addr = a_addr + kRowBytes;
          const bool second = kb >= nkx;  // accumulating Q
          const uint32_t d_tmem = tmem_base + (uint32_t)acc * 256 + (second ? 128u : 0u);
          const int kk = second ? kb - nkx : kb;
#pragma unroll
          for (int k16 = 0; k16 < kKF / 16; ++k16) {
            const uint64_t a_desc = make_sdesc_sw128(a_addr + k16 * 32, 16, 1024);
            const uint64_t b_desc = make_sdesc_sw128(b_addr + k16 * 32, 16, 1024);
            mma_bf16_pair(d_tmem, a_desc, b_desc, idesc, (kk | k16) != 0);
          }
          mma_commit_pair(empty_bar(stage));
          if (++stage == kStages) { stage = 0; phase ^= 1u; }
        }
        if (!ok) break;
        mma_commit_pair(accfull_bar(acc));
        if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
      }
    }
  } else {
    const int q = warp & 3, row = q * 32 + lane, g0 = (warp - 2) / 4 * kGroups;
    const uint32_t accempty_at_leader = map_to_cta(accempty_bar(0), 0);
    int acc = 0;
    uint32_t acc_phase = 0;
    for (Units u(p); u.more(); u.next()) {
      int I, J;
      u.get(I, J);
      I = 2 * I + (int)rank;  // this CTA's row tile; below the diagonal it has nothing to add
      const bool diag = I == J;
      // sequence of this thread's row token and of every column token (clamped past the end; those rows and columns are zero
      // in P and Q)
      const int row_seq = __ldg(p.tokseq + min((int64_t)I * kTT + row, p.T - 1));
      auto col_seq = [&](int g) { return __ldg(p.tokseq + min((int64_t)J * kTT + g * 32 + lane, p.T - 1)); };
      int cs = col_seq(g0);  // sequence of column token 32 g + lane
      if (!mbar_wait_pair(accfull_bar(acc), acc_phase, abort_flag, peer_abort, p.info, kIdGram)) break;
      tc_fence_after_sync();
      if (I <= J) {
        const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)acc * 256;
        const RowSegments rows = row_segments(row_seq, (long long)p.B * p.B, p.info);
        int cur = __shfl_sync(0xffffffffu, cs, 0);
        float wseg = row_seq == cur ? 2.f : 1.f, run = 0.f;
#pragma unroll 1
        for (int g = g0; g < g0 + kGroups; ++g) {
          const int cs_next = g + 1 < g0 + kGroups ? col_seq(g + 1) : 0;
          uint32_t pv[32], qv[32];
          tmem_ld32(taddr + g * 32, pv);
          tmem_ld32(taddr + 128 + g * 32, qv);
          tmem_ld_wait();
          gram_group<true>(pv, qv, cs, g * 32, row, diag, rows, p.K, p.B, cur, wseg, run);
          cs = cs_next;
        }
        flush_rows(p.K, p.B, rows, cur, run);
      }
      tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive_remote(accempty_at_leader + 8u * acc);
      if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
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
  CUtensorMap map[4];  // rows of X, rows of dY, columns of X, columns of dY
  for (int k = 0; k < 4; ++k) {
    const uint64_t d = k & 1 ? d_out : d_in;
    isopo_status s = make_map_2d_bf16(&map[k], k & 1 ? dY : X, (uint64_t)T, d, d, 64, k < 2 ? kTT : kTT / 2);
    if (s != ISOPO_OK) return s;
  }
  int dev = 0, sms = 0;
  ISOPO_CUDA_TRY(cudaGetDevice(&dev));
  ISOPO_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  ISOPO_CUDA_TRY(cudaFuncSetAttribute(k_bf16_gram_pair, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes));
  GramPairParams p{tokseq, K, T, B, (int)((T + kTT - 1) / kTT), (int)((T + 2 * kTT - 1) / (2 * kTT)), d_in, d_out, 0, info};
  const long long units = (long long)p.nblocks * (p.nblocks + 1);
  const int pairs = (int)std::min<long long>(units, sms / 2);
  p.strip = gram_strip_width(2.0 * 2 * kTT * (d_in + d_out), (pairs + 1) / 2);
  {
    LaunchScope scope(kIdGram, st);
    launch(k_bf16_gram_pair, 2 * pairs, kThreads, kSmemBytes, st, map[0], map[1], map[2], map[3], p);
  }
  ISOPO_CUDA_TRY(cudaGetLastError());
  return mirror_upper(K, B, st);
}

}  // namespace isopo
