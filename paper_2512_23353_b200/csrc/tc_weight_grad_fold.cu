// Stand-alone weight gradient dW = sum_i c_i G_i = (c_seq(t) dY)^T X (Alg. 1: "grad += advantages *
// rescaled gradient"; Sec. 3 display v = J^T c) with the per-sequence coefficient folded into the
// accumulator drain: no scaled copy of an operand is ever written.
//
// dW is a sum over sequences of c_i times a plain product dY_i^T X_i.  A pair of CTAs (cluster of two,
// tcgen05.mma.cta_group::2, 256 x 256 tiles, both operands token-major = "MN-major") takes a work unit
// (tile of dW, chunk of tokens) and walks the chunk one SEGMENT at a time, a segment being a maximal
// run of the chunk's tokens that belong to one sequence.  Every segment is accumulated from zero in
// one of two tensor-memory accumulators; when its last MMA has completed, the epilogue warps read the
// accumulator, multiply by the sequence's coefficient and add into a running sum that lives in
// REGISTERS (8 warps x 32 lanes x 128 columns = the CTA's 128 x 256 half of the tile) while the MMA
// thread is already filling the other accumulator with the next segment.  At the end of the unit
// the running sum is added into dW (float32 additions: the token chunks of one tile meet there), as boxes of 32 rows that TMA adds
// from shared memory: rows of 64 or 128 bytes at a time.  With red.v4 from the registers every instruction touched 32 rows, 16
// bytes of each: 1000 tokens, 896 x 896 14.7 -> 12.9 us, 40,706 66.8 -> 63.5, 9000 tokens, 1536 x 1536 39.3 -> 37.3; kPlain, 10,533
// tokens, 896 x 896 31.4 -> 29.7, 4864 x 896 82.1 -> 78.1.
// The tile never leaves the SM between segments, so against the pre-scaled-operand GEMM this saves one
// pass over the narrower operand (read + write) and its launch.
//
//   warp 0          TMA producer; both CTAs' copies complete on the barrier in CTA 0
//   warp 1, CTA 0   MMA issuer (one elected thread)
//   warps 2-9       epilogue: warp w reads TMEM lanes 32 (w mod 4) .. +31, columns 128 ((w - 2) / 4) .. +127
//   warp 10         zeroes the dY rows past the end of a segment in its last slab
//
// kPlain: the same pipeline as a plain GEMM dW += dY^T X (one operand already scaled): a piece of work is one segment with
// coefficient one.  It serves token counts for which the (256 x 512 block, slab) units of tc_weight_grad_pair.cu come out
// in rounds that are nearly empty: here the stages of all tiles, tile after tile, are cut into one equal run per pair
// ("stream K"), so a pair has about the same work whatever the shape, at the price of one or two drains more.
//
// Barriers are those of tc_seq_grad_pair.cu with "unit" read as "segment".  Every wait is bounded; a
// CTA that gives up raises the abort flag of both CTAs, and both meet at a cluster barrier before
// tensor memory is released.
#include <algorithm>

#include "tc_common.cuh"

namespace isopo {

namespace {

using namespace tc;

constexpr int kKB = 64;                              // tokens per pipeline stage
constexpr int kStages = 6;
constexpr int kHalf = 128;                           // operand columns staged per CTA (both operands)
constexpr int kChunkBytes = kKB * 128;               // one [kKB tokens][64 columns] box
constexpr int kOperandBytes = 2 * kChunkBytes;       // this CTA's half of dY or of X for one stage
constexpr int kStageBytes = 2 * kOperandBytes;
constexpr int kMaxSeqs = 2048;                       // sequences whose extents and coefficients are staged in shared memory
constexpr int kOffBytes = (kMaxSeqs + 1 + 63) / 64 * 64 * 4;
constexpr int kEpiWarps = 8;
template <bool kPlain>  // what an epilogue warp passes to dW at a time: 32 rows of 32 or 16 columns
constexpr int kBoxBytes = kPlain ? 4096 : 2048;
template <bool kPlain>
constexpr int kSmemBytes = kStages * kStageBytes + 1024 /*alignment slack*/ + 1024 /*barriers*/ + kEpiWarps * kBoxBytes<kPlain> + (kPlain ? 0 : kOffBytes + kMaxSeqs * 4);
constexpr int kThreads = 32 * (2 + kEpiWarps + 1);
constexpr uint32_t kTmemCols = 512;                  // two 256-column float32 accumulators
constexpr int kPairN = 256;
constexpr int kUnitOverhead = 6;                     // a unit's pipeline fill and flush, in stages (host cost model)
static_assert(kSmemBytes<true> <= 227 * 1024 && kSmemBytes<false> <= 227 * 1024, "shared memory");

struct FoldParams {
  const int64_t* off;    // [B + 1] token offsets
  const float* coeffs;   // [B]
  int64_t T, chunk;      // tokens per work unit (a multiple of kKB)
  int nchunks, B, d_in, d_out;
  int ptiles_m, tiles_n;  // 256-row and 256-column tiles of dW
  int group_m;            // tile rows per group of the tile order (see pair_tile)
  int32_t* info;
  int kblocks;            // kPlain: stages of one tile; a pair's run is `run` stages of ptiles * kblocks
  long long run;
  int beta;               // kPlain, 0: a tile that one pair sums alone is written, not added to
};

// Tiles are visited in groups of `group_m` rows, row index fastest inside a group, so that the pairs
// running at one time share about group_m row blocks of dY and npairs / group_m column blocks of X.
__device__ __forceinline__ void pair_tile(int pt, const FoldParams& p, int& ptm, int& tn) {
  const int per_group = p.group_m * p.tiles_n;
  const int first = (pt / per_group) * p.group_m, in_group = pt % per_group;
  const int gm = min(p.group_m, p.ptiles_m - first);
  ptm = first + in_group % gm;
  tn = in_group / gm;
}

// Columns of tile column tn that exist, in the 32-column steps of a 2-CTA MMA (see tc_seq_grad_pair.cu).
__device__ __forceinline__ int tile_cols(const FoldParams& p, int tn) { return min(kPairN, (p.d_in - tn * kPairN + 31) & ~31); }

// The pieces of work of one pair, identical in every role: (tile, tokens t0 .. t1 - 1).
template <bool kPlain>
struct Pieces {
  long long at, end, step;
  int ptiles;
  __device__ __forceinline__ Pieces(const FoldParams& p, long long pair_id, long long npairs) : ptiles(p.ptiles_m * p.tiles_n) {
    if (kPlain) {
      at = pair_id * p.run;
      end = min(at + p.run, (long long)ptiles * p.kblocks);
      step = 0;
    } else {
      at = pair_id;
      end = (long long)p.nchunks * ptiles;
      step = npairs;
    }
  }
  __device__ __forceinline__ bool next(const FoldParams& p, int& tile, int& t0, int& t1) {
    if (at >= end) return false;
    if (kPlain) {
      tile = (int)(at / p.kblocks);
      const int kb0 = (int)(at - (long long)tile * p.kblocks);
      const int kb1 = (int)min((long long)p.kblocks, kb0 + (end - at));
      t0 = kb0 * kKB;
      t1 = (int)min(p.T, (int64_t)kb1 * kKB);
      at += kb1 - kb0;
    } else {  // chunk * ptiles + tile: the pairs running at one time read the same tokens out of L2
      const int64_t a = (at / ptiles) * p.chunk;
      tile = (int)(at % ptiles);
      t0 = (int)a;
      t1 = (int)min(p.T, a + p.chunk);
      at += step;
    }
    return true;
  }
};

// Shape of one segment's token loop, identical in every role.
struct SegShape {
  int nkb;         // slabs
  int tail_n16;    // 16-token MMA steps of the last slab
  int tail_valid;  // token rows of the last slab that belong to the segment
  bool fix;        // the last step holds rows of the next segment
};
template <bool kPlain>
__device__ __forceinline__ SegShape seg_shape(int len) {
  SegShape s;
  s.nkb = (len + kKB - 1) / kKB;
  s.tail_valid = len - (s.nkb - 1) * kKB;
  s.tail_n16 = (s.tail_valid + 15) >> 4;
  s.fix = !kPlain && s.tail_valid < s.tail_n16 * 16;  // kPlain: behind a piece that ends inside a step there are no tokens
  return s;
}

// Walks the segments of the token range [t, t_end): sequence i holds tokens off[i] .. off[i+1]-1 (kPlain: one segment).
template <bool kPlain>
struct SegWalk {
  const int* off;
  int t, t_end, i;
  __device__ __forceinline__ SegWalk(const int* off32, int B, int t0, int t1) : off(off32), t(t0), t_end(t1) {
    i = 0;
    if (kPlain) return;
    int lo = 0, hi = B;  // invariant: off[lo] <= t0 < off[hi]
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (off[mid] <= t0) lo = mid; else hi = mid;
    }
    i = lo;
  }
  __device__ __forceinline__ bool done() const { return t >= t_end; }
  __device__ __forceinline__ int len() const { return (kPlain ? t_end : min(off[i + 1], t_end)) - t; }
  __device__ __forceinline__ void next() { t += len(); ++i; }
};

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}

template <bool kPlain>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
k_bf16_weight_grad_fold(const __grid_constant__ CUtensorMap mapY, const __grid_constant__ CUtensorMap mapX,
                        const __grid_constant__ CUtensorMap mapW, FoldParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t smem_base = smem_u32(smem);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kStages * kStageBytes);
  const uint32_t bar0 = smem_u32(bars);
  auto full_bar = [&](int s) { return bar0 + 8u * s; };                          // used in CTA 0
  auto empty_bar = [&](int s) { return bar0 + 8u * (kStages + s); };             // both CTAs
  auto tail_bar = [&](int s) { return bar0 + 8u * (2 * kStages + s); };          // both CTAs
  auto fixed_bar = [&](int s) { return bar0 + 8u * (3 * kStages + s); };         // used in CTA 0
  auto accfull_bar = [&](int b) { return bar0 + 8u * (4 * kStages + b); };       // both CTAs
  auto accempty_bar = [&](int b) { return bar0 + 8u * (4 * kStages + 2 + b); };  // used in CTA 0
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 4 * kStages + 4);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  // offsets (as 32-bit token indices) and coefficients, read once: the roles look them up at every
  // segment, and a global load there would stall the MMA thread for longer than its queue of MMAs lasts
  int* s_off = reinterpret_cast<int*>(smem + kStages * kStageBytes + 1024 + kEpiWarps * kBoxBytes<kPlain>);
  float* s_coef = reinterpret_cast<float*>(s_off + kOffBytes / 4);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();  // 0 issues the MMAs
  const uint32_t peer_abort = map_to_cta(smem_u32(const_cast<int*>(abort_flag)), rank ^ 1u);
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
      mbar_init(tail_bar(s), 1);
      mbar_init(fixed_bar(s), 2);
    }
    for (int b = 0; b < 2; ++b) { mbar_init(accfull_bar(b), 1); mbar_init(accempty_bar(b), 2 * kEpiWarps); }
    *abort_flag = 0;
    fence_barrier_init();
  }
  if (warp == 1) tmem_alloc_pair(smem_u32(tmem_slot), kTmemCols);
  pdl_begin();
  if (!kPlain) {
    for (int k = threadIdx.x; k <= p.B; k += kThreads) s_off[k] = (int)p.off[k];
    for (int k = threadIdx.x; k < p.B; k += kThreads) s_coef[k] = p.coeffs[k];
  }
  tc_fence_before_sync();
  __syncthreads();
  __syncwarp();
  cluster_sync_all();  // the peer's barriers exist before anything can arrive on them
  tc_fence_after_sync();
  const uint32_t tmem_base = *tmem_slot;

  const long long pair_id = blockIdx.x >> 1, npairs = gridDim.x >> 1;
  Pieces<kPlain> work(p, pair_id, npairs);
  int tile, t0, t1;

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer (both CTAs)
    if (elect_one()) {
      prefetch_tensormap(&mapY);
      prefetch_tensormap(&mapX);
      const uint32_t full_at_leader = map_to_cta(full_bar(0), 0);
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      while (ok && work.next(p, tile, t0, t1)) {
        int ptm, tn;
        pair_tile(tile, p, ptm, tn);
        const int ycol = (2 * ptm + (int)rank) * kHalf, half_cols = tile_cols(p, tn) >> 1;
        const int xcol = tn * kPairN + (int)rank * half_cols;
        const bool two = half_cols > 64;  // 64-column boxes of X per CTA
        const uint32_t x_bytes = two ? kOperandBytes : kChunkBytes;
        for (SegWalk<kPlain> w(s_off, p.B, t0, t1); !w.done() && ok; w.next()) {
          const SegShape ss = seg_shape<kPlain>(w.len());
          for (int kb = 0; kb < ss.nkb; ++kb) {
            if (!(ok = mbar_wait_pair(empty_bar(stage), phase ^ 1u, abort_flag, peer_abort, p.info, kIdWeightGrad))) break;
            const uint32_t a_dst = smem_base + stage * kStageBytes, b_dst = a_dst + kOperandBytes;
            const int y = w.t + kb * kKB;  // rows past T and columns past the matrix read as zero
            const bool own_tail = ss.fix && kb == ss.nkb - 1;  // dY goes to this CTA's tail barrier
            if (own_tail) mbar_arrive_expect_tx(tail_bar(stage), kOperandBytes);
            if (rank == 0) mbar_arrive_expect_tx(full_bar(stage), 2 * x_bytes + (own_tail ? 0 : 2 * kOperandBytes));
            const uint32_t fb = full_at_leader + 8u * stage;
#pragma unroll
            for (int c = 0; c < 2; ++c) {
              if (own_tail) tma_load_2d(a_dst + c * kChunkBytes, &mapY, ycol + c * 64, y, tail_bar(stage));
              else tma_load_2d_pair(a_dst + c * kChunkBytes, &mapY, ycol + c * 64, y, fb);
              if (c == 0 || two) tma_load_2d_pair(b_dst + c * kChunkBytes, &mapX, xcol + c * 64, y, fb);
            }
            if (++stage == kStages) { stage = 0; phase ^= 1u; }
          }
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer (one thread of CTA 0)
    if (rank == 0 && elect_one()) {
      int stage = 0, acc = 0;
      uint32_t phase = 0, acc_phase = 0, fixed_phase = 0;  // fixed_phase: one bit per stage
      bool ok = true;
      while (ok && work.next(p, tile, t0, t1)) {
        int ptm, tn;
        pair_tile(tile, p, ptm, tn);
        const uint32_t idesc = make_idesc_bf16(256, tile_cols(p, tn), /*a_mn=*/true, /*b_mn=*/true);
        for (SegWalk<kPlain> w(s_off, p.B, t0, t1); !w.done() && ok; w.next()) {
          const SegShape ss = seg_shape<kPlain>(w.len());
          if (!(ok = mbar_wait_pair(accempty_bar(acc), acc_phase ^ 1u, abort_flag, peer_abort, p.info, kIdWeightGrad))) break;
          tc_fence_after_sync();
          const uint32_t d_tmem = tmem_base + (uint32_t)acc * kPairN;
          for (int kb = 0; kb < ss.nkb; ++kb) {
            const bool last = kb == ss.nkb - 1;
            if (!(ok = mbar_wait_pair(full_bar(stage), phase, abort_flag, peer_abort, p.info, kIdWeightGrad))) break;
            if (last && ss.fix) {
              // both CTAs' dY halves of this slab have landed and their stray rows are zero
              if (!(ok = mbar_wait_pair(fixed_bar(stage), (fixed_phase >> stage) & 1u, abort_flag, peer_abort, p.info,
                                        kIdWeightGrad)))
                break;
              fixed_phase ^= 1u << stage;
            }
            tc_fence_after_sync();
            const uint32_t a_addr = smem_base + stage * kStageBytes, b_addr = a_addr + kOperandBytes;
            const int n16 = last ? ss.tail_n16 : kKB / 16;
            for (int k16 = 0; k16 < n16; ++k16) {
              const uint64_t a_desc = make_sdesc_sw128(a_addr + k16 * 2048, kChunkBytes, 1024);
              const uint64_t b_desc = make_sdesc_sw128(b_addr + k16 * 2048, kChunkBytes, 1024);
              mma_bf16_pair(d_tmem, a_desc, b_desc, idesc, (kb | k16) != 0);
            }
            mma_commit_pair(empty_bar(stage));  // frees the stage in both CTAs once these MMAs have read it
            if (++stage == kStages) { stage = 0; phase ^= 1u; }
          }
          if (!ok) break;
          mma_commit_pair(accfull_bar(acc));
          if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
        }
      }
    }
  } else if (warp < 2 + kEpiWarps) {
    // ------------------------------------------------------------------ epilogue (warps 2..9, both CTAs)
    const int q = warp & 3;            // TMEM lane quarter this warp may read
    const int h = (warp - 2) >> 2;     // column half of the tile
    const uint32_t accempty_at_leader = map_to_cta(accempty_bar(0), 0);
    int acc = 0;
    uint32_t acc_phase = 0;
    bool ok = true;
    const uint32_t box = smem_base + kStages * kStageBytes + 1024 + (warp - 2) * kBoxBytes<kPlain>;
    const bool issuer = elect_one();
    if (kPlain) {
      // A piece of work is one segment: from tensor memory straight to dW.  The loop stays rolled: its code is fetched anew in every
      // launch and runs once or twice (unrolled, with the sums in registers as below, 1000 tokens of 896 x 896 took 18 us, not 15).
      while (work.next(p, tile, t0, t1)) {
        int ptm, tn;
        pair_tile(tile, p, ptm, tn);
        const int m = (2 * ptm + (int)rank) * kHalf + q * 32, n0 = tn * kPairN + h * 128;
        const bool store = t0 == 0 && t1 == (int)p.T && !p.beta;  // the whole of this tile, nobody else's
        if (!mbar_wait_pair(accfull_bar(acc), acc_phase, abort_flag, peer_abort, p.info, kIdWeightGrad)) break;
        tc_fence_after_sync();
        const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * kPairN + h * 128);
#pragma unroll 1
        for (int jc = 0; jc < 4; ++jc) {
          uint32_t r[32];
          tmem_ld32(taddr + jc * 32, r);
          if (issuer) bulk_wait_read<0>();
          __syncwarp();
          tmem_ld_wait();
          box_row(box, lane, r);
          fence_proxy_async_smem();
          __syncwarp();
          if (issuer && m < p.d_out && n0 + jc * 32 < p.d_in) {
            if (store) tma_store_2d(&mapW, n0 + jc * 32, m, box);
            else tma_add_2d(&mapW, n0 + jc * 32, m, box);
            bulk_commit();
          }
        }
        tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive_remote(accempty_at_leader + 8u * acc);
        if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
      }
    } else {
      float sum[128];
#pragma unroll
      for (int e = 0; e < 128; ++e) sum[e] = 0.f;
      while (ok && work.next(p, tile, t0, t1)) {
        int ptm, tn;
        pair_tile(tile, p, ptm, tn);
        for (SegWalk<kPlain> w(s_off, p.B, t0, t1); !w.done(); w.next()) {
          const float c = ISOPO_IN_RANGE(w.i, p.B, p.info, kIdWeightGrad) ? s_coef[w.i] : 0.f;
          if (!(ok = mbar_wait_pair(accfull_bar(acc), acc_phase, abort_flag, peer_abort, p.info, kIdWeightGrad))) break;
          tc_fence_after_sync();
          const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * kPairN + h * 128);
#pragma unroll
          for (int jc = 0; jc < 8; ++jc) {
            uint32_t r[16];
            tmem_ld16(taddr + jc * 16, r);
            tmem_ld_wait();
#pragma unroll
            for (int e = 0; e < 16; ++e) sum[jc * 16 + e] = fmaf(c, __uint_as_float(r[e]), sum[jc * 16 + e]);
          }
          tc_fence_before_sync();
          __syncwarp();
          if (lane == 0) mbar_arrive_remote(accempty_at_leader + 8u * acc);
          if (++acc == 2) { acc = 0; acc_phase ^= 1u; }
        }
        if (!ok) break;
        // the unit's share of this tile: dW[m .., n0 .. n0 + 127] += sum, 16 columns at a time
        const int m = (2 * ptm + (int)rank) * kHalf + q * 32, n0 = tn * kPairN + h * 128;
#pragma unroll
        for (int jc = 0; jc < 8; ++jc) {
          if (issuer) bulk_wait_read<0>();
          __syncwarp();
#pragma unroll
          for (int v = 0; v < 4; ++v)
            asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(box + lane * 64 + ((v ^ ((lane >> 1) & 3)) << 4)),
                         "f"(sum[jc * 16 + 4 * v]), "f"(sum[jc * 16 + 4 * v + 1]), "f"(sum[jc * 16 + 4 * v + 2]), "f"(sum[jc * 16 + 4 * v + 3]) : "memory");
          fence_proxy_async_smem();
          __syncwarp();
          if (issuer && m < p.d_out && n0 + jc * 16 < p.d_in) {
            tma_add_2d(&mapW, n0 + jc * 16, m, box);
            bulk_commit();
          }
        }
#pragma unroll
        for (int e = 0; e < 128; ++e) sum[e] = 0.f;
      }
    }
    if (issuer) bulk_wait_read<0>();
  } else {
    // ------------------------------------------------------------------ tail warp (warp 10, both CTAs)
    // tail[s] is used only for last slabs that need the fix, so its phase is counted per stage; it
    // cannot run ahead: the stage is not reloaded before the MMA thread has passed fixed[s].
    const uint32_t fixed_at_leader = map_to_cta(fixed_bar(0), 0);
    int stage = 0;
    uint32_t tail_phase = 0;  // one bit per stage
    bool ok = true;
    while (ok && work.next(p, tile, t0, t1)) {
      for (SegWalk<kPlain> w(s_off, p.B, t0, t1); !w.done(); w.next()) {
        const SegShape ss = seg_shape<kPlain>(w.len());
        const int ts = (stage + ss.nkb - 1) % kStages;  // ring position of the last slab
        if (ss.fix) {
          if (!(ok = mbar_wait_pair(tail_bar(ts), (tail_phase >> ts) & 1u, abort_flag, peer_abort, p.info, kIdWeightGrad))) break;
          tail_phase ^= 1u << ts;
          // rows [tail_valid, tail_n16*16) hold the next segment's tokens
          const int nbytes = (ss.tail_n16 * 16 - ss.tail_valid) * 128;
          const uint32_t a_addr = smem_base + ts * kStageBytes;
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            const uint32_t base = a_addr + c * kChunkBytes + ss.tail_valid * 128;
            for (int o = lane * 16; o < nbytes; o += 32 * 16)
              asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(base + o), "r"(0u) : "memory");
          }
          fence_proxy_async_smem();
          __syncwarp();
          // the zeroed rows are in this CTA's shared memory and only this CTA's tensor core reads
          // them; the arrival (CTA scope) merely tells the MMA thread that they are there
          if (lane == 0) mbar_arrive_remote(fixed_at_leader + 8u * ts);
        }
        stage = (ts + 1) % kStages;
      }
    }
  }

  // ---------------------------------------------------------------------- teardown
  if (*abort_flag) __nanosleep(100000);  // let TMA copies already in flight land before the CTA exits
  tc_fence_before_sync();
  __syncthreads();
  __syncwarp();
  cluster_sync_all();  // neither CTA leaves (or frees tensor memory) while the other may still use it
  if (warp == 1) tmem_dealloc_pair(tmem_base, kTmemCols);
}

}  // namespace

// Where this kernel is the faster route (measured against the pre-scaled-operand GEMM of
// tc_weight_grad_pair.cu, interleaved on one B200 under its power cap): layers whose wider side is at
// most 2048 (the scaling pass there costs 10-25 % of the GEMM; q/o 1536 x 1536: 1.63-1.80 against
// 1.80-1.92 ms, 896 x 896: 0.068 against 0.083 ms).  On wider layers the other kernel's 256 x 512 blocks
// move a quarter fewer operand bytes from L2 per flop, which under the power cap outweighs its extra
// pass (8960 x 1536: 7.0-8.5 against 7.9-9.1 ms; 18944 x 3584: 34-40 against 37-48 ms).
bool bf16_weight_grad_fold_applies(int64_t T, int d_in, int d_out, int B) {
  // segments long enough that the drain per segment stays hidden
  return std::max(d_in, d_out) <= 2048 && B <= kMaxSeqs && T >= (int64_t)B * 96 &&
         T < ((int64_t)1 << 31) - 4096;
}

// Pairs of CTAs of the kernel with segments that can be resident at once.
static isopo_status resident_pairs(int* pairs) {
  int dev = 0, sms = 0;
  ISOPO_CUDA_TRY(cudaGetDevice(&dev));
  ISOPO_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  ISOPO_CUDA_TRY(cudaFuncSetAttribute(k_bf16_weight_grad_fold<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes<false>));
  static int resident[64] = {};
  if (dev < 0 || dev >= 64) return ISOPO_ERR_UNSUPPORTED;
  if (resident[dev] == 0) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * (unsigned)(sms / 2));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kSmemBytes<false>;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = 2; attr.val.clusterDim.y = 1; attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    int n = 0;
    ISOPO_CUDA_TRY(cudaOccupancyMaxActiveClusters(&n, k_bf16_weight_grad_fold<false>, &cfg));
    if (n < 1) return ISOPO_ERR_UNSUPPORTED;
    resident[dev] = std::min(n, sms / 2);
  }
  *pairs = resident[dev];
  return ISOPO_OK;
}

static isopo_status make_fold_maps(CUtensorMap* mapY, CUtensorMap* mapX, CUtensorMap* mapW, const void* X, int ldx, const void* dY, int ldy, float* dW,
                                   int64_t T, int d_in, int d_out, uint32_t box_cols) {
  isopo_status s = make_map_2d_f32(mapW, dW, (uint64_t)d_out, (uint64_t)d_in, box_cols);
  if (s != ISOPO_OK) return s;
  s = make_map_2d_bf16(mapY, dY, (uint64_t)T, (uint64_t)d_out, (uint64_t)ldy, 64, kKB);
  return s != ISOPO_OK ? s : make_map_2d_bf16(mapX, X, (uint64_t)T, (uint64_t)d_in, (uint64_t)ldx, 64, kKB);
}

static void set_group(FoldParams* p, int npairs) {
  int g = 1;
  while ((g + 1) * (g + 1) <= npairs) ++g;  // about sqrt(npairs) rows by sqrt(npairs) columns of tiles in flight
  p->group_m = std::max(1, std::min(g, p->ptiles_m));
}

// Tiles whose sums one pair holds alone are written without a clear ahead of them and without a read of what is there: where a
// tile has few stages, whole tiles per pair; where it has many, equal runs of stages, whose ends meet other runs in dW.
// All in us, runs / whole tiles: 169 tokens, 3584 x 10752 140 / 44 (clear, then additions to 154 MB, against one pass of stores:
// 3.5 TB/s), 3584 x 3584 41 / 18; 1097, 2560 x 10240 118 / 59; 2925, 2560 x 12928 204 / 162; 300, 896 x 896 12.5 / 10.2.
constexpr int kStoreStages = 8;  // stages that writing a tile takes at least, beside the MMAs of the next
PlainPlan plan_weight_grad_plain(int64_t T, int d_in, int d_out, bool add, int pairs) {
  PlainPlan plan{};
  const long long ptiles = (long long)((d_out + 2 * kHalf - 1) / (2 * kHalf)) * ((d_in + kPairN - 1) / kPairN);
  const long long kblocks = (T + kKB - 1) / kKB, stages = ptiles * kblocks;
  // no shorter runs than a drain takes
  plan.run = std::max<long long>((stages + pairs - 1) / pairs, std::min<long long>(kUnitOverhead, kblocks));
  plan.cost = plan.run + (plan.run / kblocks + 2) * kUnitOverhead;  // a run touches up to run / kblocks + 2 tiles
  const long long tiles = (ptiles + pairs - 1) / pairs, whole = tiles * std::max<long long>(kblocks, kStoreStages) + kUnitOverhead;
  if (whole <= plan.cost) { plan.run = tiles * kblocks; plan.cost = whole; }
  plan.clear = !add && plan.run % kblocks != 0;
  return plan;
}

isopo_status bf16_weight_grad_plain(const void* X, int ldx, const void* dY, int ldy, int64_t T, int d_in, int d_out, const PlainPlan& plan, bool add,
                                    float* dW, int32_t* info, cudaStream_t st) {
  ISOPO_CUDA_TRY(cudaFuncSetAttribute(k_bf16_weight_grad_fold<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes<true>));
  isopo_status s;
  CUtensorMap mapY, mapX, mapW;
  if ((s = make_fold_maps(&mapY, &mapX, &mapW, X, ldx, dY, ldy, dW, T, d_in, d_out, 32)) != ISOPO_OK) return s;
  FoldParams p{};
  p.T = T; p.d_in = d_in; p.d_out = d_out; p.info = info; p.beta = add;
  p.ptiles_m = ((d_out + kHalf - 1) / kHalf + 1) / 2;
  p.tiles_n = (d_in + kPairN - 1) / kPairN;
  p.kblocks = (int)((T + kKB - 1) / kKB);
  p.run = plan.run;
  const long long stages = (long long)p.ptiles_m * p.tiles_n * p.kblocks;
  const int npairs = (int)((stages + p.run - 1) / p.run);
  set_group(&p, npairs);
  {
    LaunchScope scope(kIdWeightGrad, st);
    launch(k_bf16_weight_grad_fold<true>, 2 * npairs, kThreads, kSmemBytes<true>, st, mapY, mapX, mapW, p);
  }
  ISOPO_CUDA_TRY(cudaGetLastError());
  return ISOPO_OK;
}

isopo_status bf16_weight_grad_fold(const void* X, const void* dY, int64_t T, int d_in, int d_out, const int64_t* off_host,
                                   int64_t* off_dev, const float* coeffs, int B, float* dW, bool add, int32_t* info, cudaStream_t st) {
  int pairs = 0;
  isopo_status s = resident_pairs(&pairs);
  if (s != ISOPO_OK) return s;
  CUtensorMap mapY, mapX, mapW;
  if ((s = make_fold_maps(&mapY, &mapX, &mapW, X, d_in, dY, d_out, dW, T, d_in, d_out, 16)) != ISOPO_OK) return s;
  FoldParams p{};
  p.off = off_dev; p.coeffs = coeffs; p.T = T; p.B = B; p.d_in = d_in; p.d_out = d_out; p.info = info;
  p.ptiles_m = ((d_out + kHalf - 1) / kHalf + 1) / 2;
  p.tiles_n = (d_in + kPairN - 1) / kPairN;
  // token chunks: the count (up to 64) whose rounds of units take least, a round costing its chunk plus the
  // unit's pipeline fill and flush; ties go to fewer chunks.  Every chunk is a whole number of stages.
  // (Chunks small enough to stay in L2 while all tiles pass over them were measured slower: the float32
  // reductions into dW and the fills grow with the chunk count, and the inputs were still read 2.6 x.)
  const long long ptiles = (long long)p.ptiles_m * p.tiles_n;
  const long long kblocks = (T + kKB - 1) / kKB;
  long long nchunks = 1, best = -1;
  for (long long n = 1; n <= std::min<long long>(64, kblocks); ++n) {
    const long long per = (kblocks + n - 1) / n, rounds = (ptiles * n + pairs - 1) / pairs;
    const long long cost = rounds * (per + kUnitOverhead);
    if (best < 0 || cost < best) { best = cost; nchunks = n; }
  }
  const long long kb_per = (kblocks + nchunks - 1) / nchunks;
  nchunks = (kblocks + kb_per - 1) / kb_per;
  p.chunk = kb_per * kKB;
  p.nchunks = (int)nchunks;
  const int npairs = (int)std::max<long long>(1, std::min<long long>(ptiles * nchunks, (long long)pairs));
  set_group(&p, npairs);
  if ((s = launch_offsets(off_host, B, off_dev, add ? Clear{} : Clear{{dW}, {(int64_t)d_in * d_out}}, st)) != ISOPO_OK) return s;
  {
    LaunchScope scope(kIdWeightGrad, st);
    launch(k_bf16_weight_grad_fold<false>, 2 * npairs, kThreads, kSmemBytes<false>, st, mapY, mapX, mapW, p);
  }
  ISOPO_CUDA_TRY(cudaGetLastError());
  return ISOPO_OK;
}

}  // namespace isopo
