// Stand-alone weight gradient dW = (c_seq(t) dY)^T X (Alg. 1: "grad += advantages * rescaled
// gradient") with 2-CTA tensor-core tiles.
//
// The coefficient of every token's sequence is applied to the NARROWER operand in one streaming pass (k_scale_rows:
// T x min(d_in, d_out) elements read and written once, round to nearest even; it also clears dW), after which the
// weight gradient is a plain GEMM over all tokens.  Scaling the landed rows in shared memory inside
// the GEMM (what the 1-CTA kernel of tc_seq_grad.cu does for small layers) was measured 15 % slower
// here: under the power cap the extra shared-memory traffic and the busy scaler warps cost more
// than the extra pass over 1/6 .. 1/35 of the operand bytes.
//
// The GEMM is the pipeline of tc_seq_grad_pair.cu with other work units: (256 x 512 block of dW, slab
// of tokens), slab-major so that the pairs running at one time read the same tokens out of L2.  The
// block is two 256 x 256 accumulators side by side that share the dY operand: all 512 columns of
// tensor memory, so a unit's epilogue is not overlapped, but a unit is a long token slab (there are
// only a few per pair).  Against one 256 x 256 tile per unit this moves 3/4 of the operand bytes
// from L2 to the SMs per flop and streams the inputs from HBM about half as often (every round of
// units re-reads its slab, and there are half as many units per slab); under the power cap both show
// up as clock.
//
//   warp 0          TMA producer; both CTAs' copies complete on the barrier in CTA 0
//   warp 1, CTA 0   MMA issuer (one elected thread), 2 x tcgen05.mma.cta_group::2 256 x 256 x 16 per step
//   warps 2-5       epilogue: TMEM -> 32 x 32 boxes in shared memory -> added into dW by TMA (token slabs of a block meet there)
//
// The additions go by boxes of 32 rows x 128 bytes, not by red.v4 (16 bytes of 32 rows an instruction): 20,000 tokens, 3584 x 8192 912
// -> 867 us, 40,000, 2136 x 968 167.7 -> 163.0; a block of one unit is written and needs no clear.
//
// Every wait is bounded; the teardown is that of tc_seq_grad_pair.cu.
#include <algorithm>

#include "tc_common.cuh"

namespace isopo {

namespace {

using namespace tc;

constexpr int kKB = 64;                              // tokens per pipeline stage
constexpr int kStages = 4;
constexpr int kHalf = 128;
constexpr int kChunkBytes = kKB * 128;           // 64 tokens x 64 columns
constexpr int kOperandBytes = 2 * kChunkBytes;   // one CTA's 128 columns of an operand
constexpr int kStageBytes = 3 * kOperandBytes;   // dY half, X half of the left tile, X half of the right tile
constexpr int kSmemBytes = kStages * kStageBytes + 1024 /*alignment slack*/ + 1024 /*barriers*/ + 4 * 8192 /*boxes of the epilogue warps*/;
constexpr int kThreads = 192;
constexpr uint32_t kTmemCols = 512;
constexpr int kPairN = 256;
constexpr int kUnitOverhead = 16;  // a unit's epilogue and pipeline fill, in 64-token stages (host cost model)
static_assert(kSmemBytes <= 227 * 1024, "shared memory");

struct FoldedPairParams {
  int64_t T, slab;  // tokens per work unit (a multiple of kKB)
  int nslabs, d_in, d_out;
  int ptiles_m, tiles_n;  // 256-row blocks of d_out; 512-column blocks of d_in
  int32_t* info;
  bool store;  // a block is one unit's alone: it is written, nothing has cleared it
};

// Columns of the left / right accumulator of block column tn that exist, in the 32-column steps of a 2-CTA MMA (see
// tc_seq_grad_pair.cu); the right one may have none.
__device__ __forceinline__ int block_cols(const FoldedPairParams& p, int tn, int right) {
  return max(0, min(kPairN, (p.d_in - (2 * tn + right) * kPairN + 31) & ~31));
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
k_bf16_weight_grad_pair(const __grid_constant__ CUtensorMap mapY, const __grid_constant__ CUtensorMap mapX,
                        const __grid_constant__ CUtensorMap mapW, FoldedPairParams p) {
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
    for (int s = 0; s < kStages; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    mbar_init(accfull_bar(0), 1);
    mbar_init(accempty_bar(0), 8);
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

  const int ptiles = p.ptiles_m * p.tiles_n;
  const long long total_units = (long long)p.nslabs * ptiles;
  const long long pair_id = blockIdx.x >> 1, npairs = gridDim.x >> 1;
  // unit u = slab * ptiles + pair tile
  auto unit_tokens = [&](long long u, int64_t& t0, int& nkb) {
    t0 = (u / ptiles) * p.slab;
    nkb = (int)((min(p.T, t0 + p.slab) - t0 + kKB - 1) / kKB);
  };

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer (both CTAs)
    if (elect_one()) {
      prefetch_tensormap(&mapY);
      prefetch_tensormap(&mapX);
      const uint32_t full_at_leader = map_to_cta(full_bar(0), 0);
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      for (long long u = pair_id; u < total_units && ok; u += npairs) {
        const int pt = (int)(u % ptiles);
        const int ptm = pt / p.tiles_n, tn = pt % p.tiles_n;
        int64_t t0;
        int nkb;
        unit_tokens(u, t0, nkb);
        const int ycol = (2 * ptm + (int)rank) * kHalf, hl = block_cols(p, tn, 0) >> 1, hr = block_cols(p, tn, 1) >> 1;
        const int xl = tn * 2 * kPairN + (int)rank * hl, xr = (tn * 2 + 1) * kPairN + (int)rank * hr;
        const uint32_t bytes = kOperandBytes + (uint32_t)(((hl + 63) >> 6) + ((hr + 63) >> 6)) * kChunkBytes;
        for (int kb = 0; kb < nkb; ++kb) {
          if (!(ok = mbar_wait_pair(empty_bar(stage), phase ^ 1u, abort_flag, peer_abort, p.info, kIdWeightGrad))) break;
          const uint32_t a_dst = smem_base + stage * kStageBytes, b_dst = a_dst + kOperandBytes;
          const int y = (int)(t0 + (int64_t)kb * kKB);  // rows past T and columns past d_in read as zero
          if (rank == 0) mbar_arrive_expect_tx(full_bar(stage), 2 * bytes);
          const uint32_t fb = full_at_leader + 8u * stage;
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            tma_load_2d_pair(a_dst + c * kChunkBytes, &mapY, ycol + c * 64, y, fb);
            if (c * 64 < hl) tma_load_2d_pair(b_dst + c * kChunkBytes, &mapX, xl + c * 64, y, fb);
            if (c * 64 < hr) tma_load_2d_pair(b_dst + kOperandBytes + c * kChunkBytes, &mapX, xr + c * 64, y, fb);
          }
          if (++stage == kStages) { stage = 0; phase ^= 1u; }
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer (one thread of CTA 0)
    if (rank == 0 && elect_one()) {
      int stage = 0;
      uint32_t phase = 0, acc_phase = 0;
      bool ok = true;
      for (long long u = pair_id; u < total_units && ok; u += npairs) {
        int64_t t0;
        int nkb;
        unit_tokens(u, t0, nkb);
        const int tn = (int)(u % ptiles) % p.tiles_n, right = block_cols(p, tn, 1);
        const uint32_t idesc = make_idesc_bf16(256, block_cols(p, tn, 0), /*a_mn=*/true, /*b_mn=*/true);
        const uint32_t idesc2 = make_idesc_bf16(256, right, /*a_mn=*/true, /*b_mn=*/true);
        if (!(ok = mbar_wait_pair(accempty_bar(0), acc_phase ^ 1u, abort_flag, peer_abort, p.info, kIdWeightGrad))) break;
        tc_fence_after_sync();
        const uint32_t d_tmem = tmem_base;
        for (int kb = 0; kb < nkb; ++kb) {
          if (!(ok = mbar_wait_pair(full_bar(stage), phase, abort_flag, peer_abort, p.info, kIdWeightGrad))) break;
          tc_fence_after_sync();
          const uint32_t a_addr = smem_base + stage * kStageBytes, b_addr = a_addr + kOperandBytes;
#pragma unroll
          for (int k16 = 0; k16 < kKB / 16; ++k16) {
            const uint64_t a_desc = make_sdesc_sw128(a_addr + k16 * 2048, kChunkBytes, 1024);
            const uint64_t b_desc = make_sdesc_sw128(b_addr + k16 * 2048, kChunkBytes, 1024);
            const uint64_t b2_desc = make_sdesc_sw128(b_addr + kOperandBytes + k16 * 2048, kChunkBytes, 1024);
            mma_bf16_pair(d_tmem, a_desc, b_desc, idesc, (kb | k16) != 0);
            if (right) mma_bf16_pair(d_tmem + kPairN, a_desc, b2_desc, idesc2, (kb | k16) != 0);
          }
          mma_commit_pair(empty_bar(stage));
          if (++stage == kStages) { stage = 0; phase ^= 1u; }
        }
        if (!ok) break;
        mma_commit_pair(accfull_bar(0));
        acc_phase ^= 1u;
      }
    }
  } else if (warp < 6) {
    // ------------------------------------------------------------------ epilogue (warps 2..5, both CTAs)
    const int q = warp & 3;
    const uint32_t accempty_at_leader = map_to_cta(accempty_bar(0), 0), boxes = smem_base + kStages * kStageBytes + 1024 + (warp - 2) * 8192;
    const bool issuer = elect_one();
    uint32_t turn = 0;  // the box that is filled next
    uint32_t acc_phase = 0;
    for (long long u = pair_id; u < total_units; u += npairs) {
      const int pt = (int)(u % ptiles);
      const int m = (2 * (pt / p.tiles_n) + (int)rank) * kHalf + q * 32, n0 = (pt % p.tiles_n) * 2 * kPairN;
      if (!mbar_wait_pair(accfull_bar(0), acc_phase, abort_flag, peer_abort, p.info, kIdWeightGrad)) break;
      tc_fence_after_sync();
      const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16);
#pragma unroll 2
      for (int jc = 0; jc < 2 * kPairN / 32 && n0 + jc * 32 < p.d_in; ++jc) {
        uint32_t r[32];
        tmem_ld32(taddr + jc * 32, r);
        if (issuer) bulk_wait_read<1>();  // of the two boxes that this warp fills in turn
        __syncwarp();
        tmem_ld_wait();
        const uint32_t box = boxes + turn * 4096;
        box_row(box, lane, r);
        fence_proxy_async_smem();
        __syncwarp();
        if (issuer && m < p.d_out) {
          if (p.store) tma_store_2d(&mapW, n0 + jc * 32, m, box);
          else tma_add_2d(&mapW, n0 + jc * 32, m, box);
        }
        if (issuer) bulk_commit();
        turn ^= 1u;
      }
      tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive_remote(accempty_at_leader);
      acc_phase ^= 1u;
    }
    if (issuer) bulk_wait_read<0>();
  }

  // ---------------------------------------------------------------------- teardown
  if (*abort_flag) __nanosleep(100000);
  tc_fence_before_sync();
  __syncthreads();
  __syncwarp();
  cluster_sync_all();
  if (warp == 1) tmem_dealloc_pair(tmem_base, kTmemCols);
}

// dst[t, :] = bf16(coeffs[sequence of t] * src[t, :]) (round to nearest even).  A warp takes a token: its first 128 16-byte pieces are on
// the way while it searches for its sequence.  HBM stream.
// kN > 0: up to kN - 1 sequences, the offsets in the arguments, so that no kernel runs ahead of this one; otherwise they are searched in
// the workspace.  46,546 tokens of 256 columns, 791 sequences: offsets and clear by a kernel of their own 2.6 + 16.7 us, so 15.7;
// 40,600 of 896, 1024 sequences 9.3 + 20.6, so 23.8.  Two tokens to a warp were slower (10,533 of 896: 6.5 -> 8.3).  Registers for six
// CTAs per SM: they wait beside the GEMM of the call before.
template <int kN>
__global__ void __launch_bounds__(256, 6) k_scale_rows(const uint4* __restrict__ src, const __grid_constant__ OffsetArgs<kN ? kN : 1> args,
                                                    const int64_t* __restrict__ off, int B, const float* __restrict__ coeffs,
                                                    int64_t T, int d8 /* columns / 8 */, uint4* __restrict__ dst, int p8 /* its pitch / 8 */,
                                                    const __grid_constant__ Clear clear) {
  __shared__ int32_t s_off[kN ? kN : 1];
  if (kN) {
    const int32_t* from = offsets_memory(args);
    for (int i = threadIdx.x; i <= B; i += blockDim.x) s_off[i] = from[i];
  }
  pdl_wait();
  __syncthreads();
  if (kN) clear_regions(clear);
  const int lane = threadIdx.x & 31;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t t = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5); t < T; t += warps) {
    const uint4* from = src + t * d8;
    uint4* to = dst + t * p8;
    uint4 v[4];
    auto load = [&](int e0) {
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (e0 + 32 * u < d8) v[u] = __ldcs(from + e0 + 32 * u);
    };
    load(lane);
    int lo = 0, hi = B;  // invariant: off[lo] <= t < off[hi]
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if ((kN ? (int64_t)s_off[mid] : off[mid]) <= t) lo = mid; else hi = mid;
    }
    const float c = __ldg(coeffs + lo);
    for (int e0 = lane; e0 < d8; e0 += 128) {
      if (e0 != lane) load(e0);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (e0 + 32 * u >= d8) continue;
        uint32_t* w = reinterpret_cast<uint32_t*>(&v[u]);
#pragma unroll
        for (int k = 0; k < 4; ++k)
          w[k] = pack_bf16x2(c * __uint_as_float(w[k] << 16), c * __uint_as_float(w[k] & 0xffff0000u));
        to[e0 + 32 * u] = v[u];
      }
    }
  }
}

}  // namespace

isopo_status bf16_weight_grad_pair(const void* X, const void* dY, int64_t T, int d_in, int d_out, const int64_t* off_host,
                                   int64_t* off_dev, const float* coeffs, int B, void* scaled, int scaled_ld, float* dW, bool add, int32_t* info,
                                   cudaStream_t st) {
  int dev = 0, sms = 0;
  ISOPO_CUDA_TRY(cudaGetDevice(&dev));
  ISOPO_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  ISOPO_CUDA_TRY(cudaFuncSetAttribute(k_bf16_weight_grad_pair, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes));
  static int resident_pairs[64] = {};
  if (dev < 0 || dev >= 64) return ISOPO_ERR_UNSUPPORTED;
  if (resident_pairs[dev] == 0) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * (unsigned)(sms / 2));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kSmemBytes;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = 2; attr.val.clusterDim.y = 1; attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    int n = 0;
    ISOPO_CUDA_TRY(cudaOccupancyMaxActiveClusters(&n, k_bf16_weight_grad_pair, &cfg));
    if (n < 1) return ISOPO_ERR_UNSUPPORTED;
    resident_pairs[dev] = std::min(n, sms / 2);
  }
  FoldedPairParams p{};
  p.T = T; p.d_in = d_in; p.d_out = d_out; p.info = info;
  p.ptiles_m = ((d_out + kHalf - 1) / kHalf + 1) / 2;
  p.tiles_n = (d_in + 2 * kPairN - 1) / (2 * kPairN);
  // token slabs: the count (up to 64) whose rounds of units take least, a round costing its slab plus the
  // unit's exposed epilogue and pipeline fill (about kUnitOverhead stages' worth); ties go to fewer slabs.  Every slab is a multiple of the stage depth.
  // (Slabs small enough for their rows to stay in L2 across the rounds were measured slower: the
  // float32 reductions into dW grow with the slab count.)
  const long long ptiles = (long long)p.ptiles_m * p.tiles_n, pairs = resident_pairs[dev];
  const long long kblocks = (T + kKB - 1) / kKB;
  long long nslabs = 1, best = -1;
  for (long long n = 1; n <= std::min<long long>(64, kblocks); ++n) {
    const long long per = (kblocks + n - 1) / n, rounds = (ptiles * n + pairs - 1) / pairs;
    const long long cost = rounds * (per + kUnitOverhead);
    if (best < 0 || cost < best) { best = cost; nslabs = n; }
  }
  // The other kernel (256 x 256 tiles, every pair the same number of stages) where these units leave the last round too
  // empty (a stage of 512 columns is two of 256) and the inputs stay in the L2: its pairs walk the tokens at different
  // places.  10,496 tokens, 896 x 4864 (121 MB) 100 -> 84 us, 4864 x 896 102 -> 74 us; 40,960 tokens, 896 x 896 (147 MB)
  // 67 -> 94 us, 35,200 tokens, 896 x 4864 (405 MB) 301 -> 445 us.
  const bool in_l2 = 2.0 * (double)T * (d_in + d_out) <= 128e6;
  const PlainPlan plan = plan_weight_grad_plain(T, d_in, d_out, add, (int)pairs);
  const bool plain = in_l2 && 10 * plan.cost < 9 * 2 * best;
  const long long kb_per = (kblocks + nslabs - 1) / nslabs;
  nslabs = (kblocks + kb_per - 1) / kb_per;
  p.slab = kb_per * kKB;
  p.nslabs = (int)nslabs;
  p.store = !add && nslabs == 1;
  const Clear clear = !add && (plain ? plan.clear : !p.store) ? Clear{{dW}, {(int64_t)d_in * d_out}} : Clear{};
  int ldx = d_in, ldy = d_out;
  {  // scale the narrower operand into `scaled`
    const bool scale_y = d_out <= d_in;
    const int d8 = (scale_y ? d_out : d_in) / 8, p8 = scaled_ld / 8;
    const uint4* src = (const uint4*)(scale_y ? dY : X);
    int64_t ctas = (T + 7) / 8;
    // One launch less (1 to 3 us of a small layer's pass).  The clear needs its share of the chip: with one CTA for every 8 of
    // 4000 tokens a 4096 x 4096 dW took 10 us longer than from a kernel of its own, hence a CTA for every 16 KB as well.
    ctas = std::max(ctas, clear.n[0] / 4096);
    const int grid = (int)std::min<int64_t>(ctas, (int64_t)sms * 16);
    auto with_args = [&](auto kernel, auto* a) {
      fill_offsets(a, off_host, B + 1);
      LaunchScope scope(kIdScaleRows, st);
      launch(kernel, grid, 256, 0, st, src, *a, off_dev, B, coeffs, T, d8, (uint4*)scaled, p8, clear);
    };
    if (B + 1 <= kArgChunk) {
      OffsetArgs<kArgChunk> a;
      with_args(k_scale_rows<kArgChunk>, &a);
    } else if (B + 1 <= kArgLarge) {
      OffsetArgs<kArgLarge> a;
      with_args(k_scale_rows<kArgLarge>, &a);
    } else {
      isopo_status s = launch_offsets(off_host, B, off_dev, clear, st);
      if (s != ISOPO_OK) return s;
      LaunchScope scope(kIdScaleRows, st);
      launch(k_scale_rows<0>, grid, 256, 0, st, src, OffsetArgs<1>{}, off_dev, B, coeffs, T, d8, (uint4*)scaled, p8, Clear{});
    }
    ISOPO_CUDA_TRY(cudaGetLastError());
    if (scale_y) { dY = scaled; ldy = 8 * p8; } else { X = scaled; ldx = 8 * p8; }
  }
  if (plain) return bf16_weight_grad_plain(X, ldx, dY, ldy, T, d_in, d_out, plan, add, dW, info, st);
  CUtensorMap mapY, mapX;
  isopo_status s = make_map_2d_bf16(&mapY, dY, (uint64_t)T, (uint64_t)d_out, (uint64_t)ldy, 64, kKB);
  if (s != ISOPO_OK) return s;
  s = make_map_2d_bf16(&mapX, X, (uint64_t)T, (uint64_t)d_in, (uint64_t)ldx, 64, kKB);
  if (s != ISOPO_OK) return s;
  CUtensorMap mapW;
  if ((s = make_map_2d_f32(&mapW, dW, (uint64_t)d_out, (uint64_t)d_in, 32)) != ISOPO_OK) return s;
  const int npairs = (int)std::max<long long>(1, std::min<long long>(ptiles * nslabs, pairs));
  {
    LaunchScope scope(kIdWeightGrad, st);
    launch(k_bf16_weight_grad_pair, 2 * npairs, kThreads, kSmemBytes, st, mapY, mapX, mapW, p);
  }
  ISOPO_CUDA_TRY(cudaGetLastError());
  return ISOPO_OK;
}

}  // namespace isopo
