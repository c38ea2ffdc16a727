// K = G_flat G_flat^T from the stored per-sequence gradients (Alg. 2 "make neural tangent kernel":
// K_ij = sum(G_i * G_j)), and dW = sum_i c_i G_i from the same store (Alg. 2 last line).
//
// k_bf16_ntk: the B <= 256 stored gradients form a [pieces][B][256] bf16 array (tc_common.cuh).  Each CTA
// takes a contiguous run of the long contraction dimension, streams [B rows] x [64 elements] boxes
// (four per piece, so a CTA walks memory front to back) through a TMA ring, and uses every box as BOTH tcgen05 operands (K-major): rows 0..127 against all rows,
// then rows 128..255 against rows 128..255 (the lower-left block is the mirror of the upper-right).
// The float32 accumulators stay in tensor memory for the whole slab and are added up once: 32 x 32 blocks of one triangle go
// through shared memory to TMA reductions into rows that a last tiny kernel completes K from.  (One float atomic per entry into
// K, every CTA in the same order, was half of the pass where the layer is not large, and 8 us of any: 10,000 tokens, 480 x 448, K pass
// of 100 sequences 24.9 -> 9.9 us, 139 23.2 -> 15.9; 896 x 128, 64 sequences 13.4 -> 7.7, 256 23.1 -> 14.7; 896 x 896, 64 25.2 -> 20.9.)
// For B <= 128 a box holds few rows that do not exist (4, 8, .. 128 >= B) but spans 64, 32, .. 2 pieces, so
// that every TMA copy still moves 32 KB (small boxes cost a fixed ~100 clocks each) and the stage is
// again 256 rows: rows 0..127 and rows 128..255 each go through ONE 128 x 128 MMA per 16 elements,
// which multiplies up to 32 pieces at once.  Only the diagonal blocks of that product (a piece
// against itself) are wanted; the epilogue adds them into K and skips the cross-piece blocks.  The
// tensor pipe does up to four times the needed work this way, but in a quarter of the instructions:
// with one 128 x 64 MMA per piece the pass was bound by the MMA issue rate (4.0 TB/s at B = 64
// against 5.4 TB/s at B = 256 on the same clock), and the pipe has time to spare in an HBM-bound pass.
// The order of the blocks inside the long contraction does not matter.
//
// k_bf16_combine: pure streaming, one 16-byte slot per lane; a warp reads 512
// contiguous bytes per sequence and the sequences of a piece back to back.
#include "tc_common.cuh"

namespace isopo {

namespace {

using namespace tc;

constexpr int kKB = 64;               // contraction elements per stage (one 128-byte row)
constexpr int kStages = 6;
constexpr int kStageBytes = 256 * 128;  // 256 rows x 128 bytes
constexpr int kSmemBytes = kStages * kStageBytes + 1024 + 256 + 1024 /* reciprocal scales of the split store */;
constexpr int kThreads = 192;
constexpr uint32_t kTmemCols = 512;

struct NtkParams {
  float* kpart;   // deterministic mode: [CTA][B * B] partial sums, plain stores; NULL: float atomics into K
  const float* scales;  // split store: s_i per sequence (the `hi` plane holds s_i G_i); the diagonal is not written here
  float* K;
  int B;
  long long nkb;  // boxes in the contraction dimension: ceil(pieces / ppb) * 4
  int32_t* info;
  int box_rows;   // rows of a piece inside a box: 4, 8, .. 256, >= B
  int ppb;        // pieces per box = 256 / box_rows
  // not NULL (up to 16 sequences, 32 with little data): the last CTA to add its share completes the other triangle and the
  // diagonal of the split store
  uint32_t* done;
  uint32_t n_active;  // CTAs with a share
  const float* kdiag;
};

// kE4m3: the operand is the `hi` plane of the split store: 128 one-byte elements per 128-byte box row (two boxes
// per piece instead of four), kind::f8f6f4 MMAs of 32 elements each - the same number of MMAs per byte, half the bytes.
// The end of it, by kSums: kFew (boxes of fewer than 32 rows) and kRows add into K or store partial sums, kBoxes adds boxes by TMA.  Each a
// kernel of its own, as their code is fetched anew in every launch and runs once.
enum NtkSums { kFew, kRows, kBoxes };
template <bool kE4m3, NtkSums kSums>
__global__ void __launch_bounds__(kThreads, 1) k_bf16_ntk(const __grid_constant__ CUtensorMap mapG, const __grid_constant__ CUtensorMap mapK, NtkParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t smem_base = smem_u32(smem);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kStages * kStageBytes);
  const uint32_t bar0 = smem_u32(bars);
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (kStages + s); };
  const uint32_t accfull_bar = bar0 + 8u * (2 * kStages);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kStages + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
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
  tc_fence_after_sync();
  const uint32_t tmem_base = *tmem_slot;

  // this CTA's slab of the contraction dimension
  const long long per = (p.nkb + gridDim.x - 1) / gridDim.x;
  const long long kb0 = (long long)blockIdx.x * per, kb1 = min(p.nkb, kb0 + per);
  const bool two = p.B > 128;                       // one piece per box, K in two row blocks
  const uint32_t stage_tx = kStageBytes;            // rows >= B and pieces past the end arrive as zeros and count
  // MMA 1: rows 0..127 against n1 rows from row 0; MMA 2: rows 128..255 against n2 rows from row 128
  const int n1 = two ? 256 : (p.box_rows == 128 ? max(16, (p.B + 15) & ~15) : 128);
  const int n2 = two ? max(16, (p.B - 128 + 15) & ~15) : n1;

  if (kb0 < kb1) {
    if (warp == 0) {
      if (elect_one()) {
        prefetch_tensormap(&mapG);
        int stage = 0;
        uint32_t phase = 0;
        for (long long kb = kb0; kb < kb1; ++kb) {
          if (!mbar_wait(empty_bar(stage), phase ^ 1u, abort_flag, p.info, kIdNtk)) break;
          mbar_arrive_expect_tx(full_bar(stage), stage_tx);
          if (kE4m3)
            tma_load_3d(smem_base + stage * kStageBytes, &mapG, (int)(kb & 1) * 128, 0, (int)(kb >> 1) * p.ppb, full_bar(stage));
          else
            tma_load_3d(smem_base + stage * kStageBytes, &mapG, (int)(kb & 3) * kKB, 0, (int)(kb >> 2) * p.ppb, full_bar(stage));
          if (++stage == kStages) { stage = 0; phase ^= 1u; }
        }
      }
    } else if (warp == 1) {
      if (elect_one()) {  // elected, not "lane 0": lets the compiler keep the MMA operands in uniform registers
        const uint32_t idesc1 = kE4m3 ? make_idesc_e4m3(128, n1) : make_idesc_bf16(128, n1, false, false);
        const uint32_t idesc2 = kE4m3 ? make_idesc_e4m3(128, n2) : make_idesc_bf16(128, n2, false, false);
        int stage = 0;
        uint32_t phase = 0;
        bool ok = true;
        for (long long kb = kb0; kb < kb1; ++kb) {
          if (!(ok = mbar_wait(full_bar(stage), phase, abort_flag, p.info, kIdNtk))) break;
          tc_fence_after_sync();
          const uint32_t base = smem_base + stage * kStageBytes;
#pragma unroll
          for (int k16 = 0; k16 < kKB / 16; ++k16) {
            const bool accum = (kb > kb0) || k16 > 0;
            const uint64_t d0 = make_sdesc_sw128(base + k16 * 32, 16, 1024);
            const uint64_t d1 = make_sdesc_sw128(base + 128 * 128 + k16 * 32, 16, 1024);
            if (kE4m3) {
              mma_e4m3(tmem_base, d0, d0, idesc1, accum);
              mma_e4m3(tmem_base + 256, d1, d1, idesc2, accum);
            } else {
              mma_bf16(tmem_base, d0, d0, idesc1, accum);
              mma_bf16(tmem_base + 256, d1, d1, idesc2, accum);
            }
          }
          mma_commit(empty_bar(stage));
          if (++stage == kStages) { stage = 0; phase ^= 1u; }
        }
        if (ok) mma_commit(accfull_bar);
      }
    } else {
      const int q = warp & 3;
      const int r = q * 32 + lane;
      // `ok` is false only after a wait ran out; every thread still reaches the named barriers below
      const bool ok = mbar_wait(accfull_bar, 0, abort_flag, p.info, kIdNtk);
      // split store: the accumulators hold s_i s_j <G_i, G_j>; 1 / s_i of every sequence goes to shared memory, and the
      // diagonal is left to the gradient GEMM's float32 sums
      float* inv_s = reinterpret_cast<float*>(smem + kStages * kStageBytes + 256);
      if (kE4m3) {
        for (int i = r; i < 256; i += 128) inv_s[i] = i < p.B ? 1.f / __ldg(p.scales + i) : 0.f;
        asm volatile("bar.sync 2, 128;" ::: "memory");
      }
      auto unscale = [&](int row, int col, float v) { return kE4m3 ? v * inv_s[row] * inv_s[col] : v; };
      if (kSums == kBoxes) {
        // Blocks of 32 columns c of the warp's 32 accumulator rows go through shared memory (the ring is idle by now), turned over so
        // that box row c holds K[c][r .. r + 31], and are added by TMA into the rows of p.acc; what the diagonal blocks have
        // above the diagonal is not read from there.  A CTA starts at a block of its own: 148 of them on one sector wait for one another.
        // Up to 128 sequences both accumulators hold sums of the same blocks, up to 64 so do warps q and q + 2: they are added up here, so
        // that an entry of K is a sum of one float32 addition per CTA (four of them had twice the error: 64 sequences 3.5e-7 against 1.8e-7).
        tc_fence_after_sync();
        constexpr int kRingBytes = kStages * kStageBytes / 4;
        const uint32_t tlane = (uint32_t)(q * 32) << 16, ring = smem_base + q * kRingBytes, partner = smem_base + (q ^ 2) * kRingBytes;
        const bool issuer = elect_one(), halves = p.box_rows == 64;
        // sequences of the warp's rows in the left accumulator (the right one: the same, or rows 128 ..), first column of their piece
        const int seq0 = two ? q * 32 : (q * 32) & (p.box_rows - 1), coff = two ? 0 : q * 32 - seq0;
        const int na = ok ? max(0, ((two ? n1 : min(p.box_rows, p.B)) - seq0 + 31) >> 5) : 0;       // blocks at and right of the diagonal
        auto send = [&](int sr, int sc, uint32_t box, const uint32_t (&v)[32]) {  // sequences of the block's first row and column
#pragma unroll
          for (int e = 0; e < 32; ++e) {
            const float x = kE4m3 ? unscale(sr + lane, sc + e, __uint_as_float(v[e])) : __uint_as_float(v[e]);
            asm volatile("st.shared.f32 [%0], %1;" ::"r"(box + e * 128 + lane * 4), "f"(x) : "memory");
          }
          fence_proxy_async_smem();
          __syncwarp();
          if (issuer) {
            tma_add_2d(&mapK, sr, sc, box);
            bulk_commit();
          }
        };
        if (two) {
          const int nb = ok ? max(0, (n2 - seq0 + 31) >> 5) : 0, n = na + nb, first = n ? blockIdx.x % n : 0;
#pragma unroll 1
          for (int k = 0; k < n; ++k) {
            const int b = first + k < n ? first + k : first + k - n;
            const bool right = b >= na;
            const int c = seq0 + (right ? b - na : b) * 32;                  // accumulator column
            const int sr = seq0 + (right ? 128 : 0), sc = c + (right ? 128 : 0);
            if (sr >= p.B || sc >= p.B) continue;
            uint32_t v[32];
            tmem_ld32(tmem_base + tlane + (right ? 256 : 0) + c, v);
            tmem_ld_wait();
            send(sr, sc, ring + k * 4096, v);
          }
        } else {
          auto load = [&](int c, uint32_t (&v)[32]) {  // accumulator column c of the piece
            uint32_t w[32];
            tmem_ld32(tmem_base + tlane + coff + c, v);
            tmem_ld32(tmem_base + tlane + 256 + coff + c, w);
            tmem_ld_wait();
#pragma unroll
            for (int e = 0; e < 32; ++e) v[e] = __float_as_uint(__uint_as_float(v[e]) + __uint_as_float(w[e]));
          };
          auto others = [&](int b) { return halves && ((b ^ (q >> 1)) & 1); };  // block b is warp q ^ 2's to send
          if (halves) {
#pragma unroll 1
            for (int b = 0; b < na; ++b) {
              if (!others(b)) continue;
              uint32_t v[32];
              load(seq0 + b * 32, v);
#pragma unroll
              for (int e = 0; e < 32; ++e) asm volatile("st.shared.b32 [%0], %1;" ::"r"(ring + b * 4096 + e * 128 + lane * 4), "r"(v[e]) : "memory");
            }
            asm volatile("bar.sync 1, 128;" ::: "memory");  // the four epilogue warps
          }
          const int first = na ? blockIdx.x % na : 0;
#pragma unroll 1
          for (int k = 0; k < na; ++k) {
            const int b = first + k < na ? first + k : first + k - na, c = seq0 + b * 32;
            if (seq0 >= p.B || c >= p.B || others(b)) continue;
            uint32_t v[32];
            load(c, v);
            if (halves) {
#pragma unroll
              for (int e = 0; e < 32; ++e) {
                float x;
                asm volatile("ld.shared.f32 %0, [%1];" : "=f"(x) : "r"(partner + b * 4096 + e * 128 + lane * 4) : "memory");
                v[e] = __float_as_uint(__uint_as_float(v[e]) + x);
              }
            }
            send(seq0, c, ring + b * 4096, v);
          }
        }
        if (issuer) bulk_wait_read<0>();
      } else {
        // deterministic mode, few sequences, no room for padded rows
        // every (CTA, entry of the lower triangle) is produced by exactly one thread, once.  Entry (r, c), c >= r, goes to
        // K[c][r]: the 32 lanes of a warp own consecutive r, so one instruction adds 128 contiguous bytes.
        float* const mine = p.kpart ? p.kpart + (size_t)blockIdx.x * p.B * p.B : nullptr;
        auto add_to_k = [&](size_t idx, float v) {
          if (mine) mine[idx] = v; else atomicAdd(&p.K[idx], v);
        };
        tc_fence_after_sync();
        const uint32_t tlane = (uint32_t)(q * 32) << 16;
        if (kSums == kRows && two && ok) {
          // block A: rows 0..127 x columns 0..255 of K; keep the upper triangle c >= r
          for (int c0 = 0; c0 < n1; c0 += 32) {
            uint32_t v[32];
            tmem_ld32(tmem_base + tlane + c0, v);
            tmem_ld_wait();
            if (r < p.B) {
#pragma unroll
              for (int e = 0; e < 32; ++e) {
                const int c = c0 + e;
                if (c >= r + (kE4m3 ? 1 : 0) && c < p.B &&
                    ISOPO_IN_RANGE((long long)c * p.B + r, (long long)p.B * p.B, p.info, kIdNtk))
                  add_to_k((size_t)c * p.B + r, unscale(r, c, __uint_as_float(v[e])));
              }
            }
          }
          // block B: rows 128..255 x columns 128..255
          const int rr = 128 + r;
          for (int c0 = 0; c0 < n2; c0 += 32) {
            uint32_t v[32];
            tmem_ld32(tmem_base + tlane + 256 + c0, v);
            tmem_ld_wait();
            if (rr < p.B) {
#pragma unroll
              for (int e = 0; e < 32; ++e) {
                const int c = 128 + c0 + e;
                if (c >= rr + (kE4m3 ? 1 : 0) && c < p.B &&
                    ISOPO_IN_RANGE((long long)c * p.B + rr, (long long)p.B * p.B, p.info, kIdNtk))
                  add_to_k((size_t)c * p.B + rr, unscale(rr, c, __uint_as_float(v[e])));
              }
            }
          }
        } else if (!two) {
          // both accumulators hold 128 / box_rows pieces side by side: row r is sequence r mod box_rows of
          // piece-group g = r / box_rows, whose columns start at g * box_rows.  Every thread leaves the sum
          // of its two accumulator rows in shared memory (the ring is idle by now); then the 128 threads
          // walk the box_rows x box_rows block together, add the groups and update K.
          const int lr = 31 - __clz(p.box_rows), rows = 1 << lr;  // box_rows is a power of two
          const int seq = r & (rows - 1), g = r >> lr, ngroups = 128 >> lr;
          // the columns that a warp reads are the same for its lanes: of fewer than 32 sequences the whole block on its diagonal
          const int coff = (q * 32) & ~(rows - 1), mine = lane & ~(rows - 1);
          const int ncol = min(rows, p.B);
          float* red = reinterpret_cast<float*>(smem);  // [group][column][sequence]
          if (ok) {
            for (int c0 = 0; c0 < ncol; c0 += 32) {
              uint32_t v0[32], v1[32];
              tmem_ld32(tmem_base + tlane + coff + c0, v0);
              tmem_ld32(tmem_base + tlane + 256 + coff + c0, v1);
              tmem_ld_wait();
              float* dst = red + ((((g << lr) + c0) << lr) + seq);
              if (kSums == kRows) {
#pragma unroll
                for (int e = 0; e < 32; ++e) dst[e << lr] = __uint_as_float(v0[e]) + __uint_as_float(v1[e]);
              } else {
#pragma unroll
                for (int e = 0; e < 32; ++e) {
                  const int c = e - mine;
                  if (c >= 0 && c < rows) dst[c << lr] = __uint_as_float(v0[e]) + __uint_as_float(v1[e]);
                }
              }
            }
          }
          asm volatile("bar.sync 1, 128;" ::: "memory");  // the four epilogue warps
          if (ok) {
            for (int idx = r; idx < (ncol << lr); idx += 128) {
              const int sq = idx & (rows - 1), c = idx >> lr;
              if (c < sq + (kE4m3 ? 1 : 0) || sq >= p.B) continue;  // one triangle of the sequences that exist
              float sum = 0.f;
              for (int h = 0; h < ngroups; ++h) sum += red[(((h << lr) + c) << lr) + sq];
              if (ISOPO_IN_RANGE((long long)c * p.B + sq, (long long)p.B * p.B, p.info, kIdNtk))
                add_to_k((size_t)c * p.B + sq, unscale(sq, c, sum));
            }
          }
          if (p.done) {
            volatile int* last = abort_flag + 1;
            __threadfence();
            asm volatile("bar.sync 1, 128;" ::: "memory");
            if (r == 0) *last = atomicAdd(p.done, 1u) == p.n_active - 1;
            asm volatile("bar.sync 1, 128;" ::: "memory");
            if (*last) {
              __threadfence();
              mirror_by_cta<false>(p.K, p.B, r, [&](int i) { return p.kdiag[i]; }, kE4m3);
            }
          }
        }
      }
    }
  }

  if (*abort_flag) __nanosleep(100000);
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem_base, kTmemCols);
}

// Deterministic mode: K[i][j] = K[j][i] = sum over the CTAs, in CTA order, of their partial entry (i, j), i >= j.
// One thread per entry of the lower triangle (its reads run along a row of every partial matrix), which also
// writes the mirrored entry.
__global__ void k_ntk_reduce(const float* __restrict__ kpart, int n_ctas, int B, float* __restrict__ K) {
  pdl_wait();
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= B * B) return;
  const int i = e / B, j = e % B;
  if (j > i) return;
  const size_t stride = (size_t)B * B;
  float s = 0.f;
  int c = 0;
  for (; c + 8 <= n_ctas; c += 8) {  // eight loads in flight; the additions keep the CTA order
    float v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = __ldcs(kpart + (c + u) * stride + e);
#pragma unroll
    for (int u = 0; u < 8; ++u) s += v[u];
  }
  for (; c < n_ctas; ++c) s += __ldcs(kpart + c * stride + e);
  K[e] = s;
  K[(size_t)j * B + i] = s;
}

// K[j][i] = K[i][j] for i < j: the triangle that a Gram kernel left out.
__global__ void k_mirror(float* __restrict__ K, int B) {
  pdl_wait();
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= B * B) return;
  const int i = e / B, j = e % B;
  if (j < i) K[e] = K[(size_t)j * B + i];
}
// K from the triangle i >= j of the K pass's sums (rows of `ld` floats).
// kdiag != NULL (split store): the diagonal comes from the gradient GEMM's float32 sums of squares
// (acc may be K itself: what of it is read is written unchanged)
__global__ void k_ntk_finish(const float* acc, int ld, float* K, int B, const float* __restrict__ kdiag) {
  pdl_wait();
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= B * B) return;
  const int i = e / B, j = e % B;
  K[e] = i == j && kdiag ? kdiag[i] : acc[(size_t)max(i, j) * ld + min(i, j)];
}

#ifndef ISOPO_COMBINE_IN_FLIGHT
#define ISOPO_COMBINE_IN_FLIGHT 16
#endif
constexpr int kCombineInFlight = ISOPO_COMBINE_IN_FLIGHT;  // 16-byte loads a thread has in flight
// dW = beta dW + sum_i c_i G_i.  HBM stream.  A warp takes the 32 slots of a piece (16 bytes = 8 elements of every G_i per
// lane) and one of kSlices shares of the sequences; the shares meet in shared memory.  One share (every lane sums all B
// sequences) is the plain stream of a wide layer; a narrow layer has too few pieces to fill the machine that way and
// splits the sequences instead (combine_slices below).  896 -> 128, one share against eight: 64 sequences 16.6 against
// 11.5 us, 256 sequences 41 against 17 us.
// kMany: kCombineInFlight loads of a lane in flight and the remainder one by one, for long sums.  Otherwise eight, the
// remainder together as well, and registers for twice the CTAs per SM, for short ones (kManySeqs).
template <int kSlices, bool kMany>
__global__ void __launch_bounds__(256, kMany ? 1 : 4) k_bf16_combine(const uint4* __restrict__ G, long long nchunks /* n_pad / 8 */,
                                                       int B, PieceGrid grid, int d_in, int d_out,
                                                       const float* __restrict__ coeffs, float* __restrict__ dW,
                                                       float beta, const WsTag* __restrict__ tag_dev, WsTag tag,
                                                       int32_t* __restrict__ info) {
  pdl_wait();
  if (!ws_tag_matches(tag_dev, tag, info)) return;  // another layer's or microbatch's gradients: touch nothing
  constexpr int kPieces = 8 / kSlices;  // pieces a block works on at a time
  constexpr int kF = kMany ? kCombineInFlight : 8;
  static_assert(kSlices == 1 || !kMany, "a share is short");
  __shared__ float sc[256];
  __shared__ float4 part[kSlices > 1 ? 8 * 64 : 1];
  for (int i = threadIdx.x; i < B; i += blockDim.x) sc[i] = coeffs[i];
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int npieces = (int)(nchunks >> 5);
  const int per = (B + kSlices - 1) / kSlices, i0 = (warp % kSlices) * per, i1 = min(B, i0 + per);
  // where a lane's 4 columns n .. n + 3 of row m go, or NULL; what is there is read ahead of the sums (a read behind them, half
  // of a sector at a time, was waited for: 40 sequences of 1536 x 4096, beta = 1, 143 us against 82)
  auto place = [&](int m, int n) -> float4* {
    if (m >= d_out || !ISOPO_IN_RANGE((long long)m * d_in + n + 3, (long long)d_out * d_in, info, kIdCombine)) return nullptr;
    return reinterpret_cast<float4*>(dW + (size_t)m * d_in + n);
  };
  auto before = [&](const float4* at) { return beta != 0.f && at ? *at : make_float4(0.f, 0.f, 0.f, 0.f); };
  auto write = [&](float4* at, float4 o, const float4& p) {
    if (beta != 0.f) { o.x += p.x; o.y += p.y; o.z += p.z; o.w += p.w; }
    if (at) *at = o;
  };
  for (int p0 = blockIdx.x * kPieces; p0 < npieces; p0 += gridDim.x * kPieces) {
    const int piece = p0 + warp / kSlices;
    const bool live = piece < npieces &&
                      ISOPO_IN_RANGE((long long)stored_slot((size_t)piece, B - 1, B, lane), nchunks * B, info, kIdCombine);
    float4 *out0 = nullptr, *out1 = nullptr;  // whole sums: the lane's row of its piece
    if (kSlices == 1 && live) {
      int m, n;
      grid.origin(piece, m, n);
      out0 = place(m + lane, n);
      out1 = place(m + lane, n + 4);
    }
    const float4 old0 = before(out0), old1 = before(out1);
    float acc[8] = {};
    const uint4* src = G + stored_slot((size_t)piece, 0, B, lane);
    const size_t stride = 32;  // slots between successive sequences of one piece
    auto add = [&](const uint4& v, float c) {
      const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        acc[2 * h] = fmaf(c, __uint_as_float(w[h] << 16), acc[2 * h]);
        acc[2 * h + 1] = fmaf(c, __uint_as_float(w[h] & 0xffff0000u), acc[2 * h + 1]);
      }
    };
    if (kSlices == 1) {
      int i = 0;
      for (; live && i + kF <= B; i += kF) {
        uint4 v[kF];
#pragma unroll
        for (int u = 0; u < kF; ++u) v[u] = __ldcs(src + (size_t)(i + u) * stride);
#pragma unroll
        for (int u = 0; u < kF; ++u) add(v[u], sc[i + u]);
      }
      if (kMany) {
        for (; live && i < B; ++i) add(__ldcs(src + (size_t)i * stride), sc[i]);
      } else if (live && i < B) {
        uint4 v[kF];
#pragma unroll
        for (int u = 0; u < kF; ++u) v[u] = i + u < B ? __ldcs(src + (size_t)(i + u) * stride) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int u = 0; u < kF; ++u) add(v[u], i + u < B ? sc[i + u] : 0.f);
      }
    } else {
      // a share is a few loads long: all of them in flight at once, the remainder too
      for (int i = i0; i < i1; i += kF) {
        uint4 v[kF];
#pragma unroll
        for (int u = 0; u < kF; ++u) v[u] = live && i + u < i1 ? __ldcs(src + (size_t)(i + u) * stride) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int u = 0; u < kF; ++u) add(v[u], i + u < i1 ? sc[i + u] : 0.f);
      }
    }
    const float4 lo = make_float4(acc[0], acc[1], acc[2], acc[3]), hi = make_float4(acc[4], acc[5], acc[6], acc[7]);
    if (kSlices == 1) {
      write(out0, lo, old0);
      write(out1, hi, old1);
    } else {
      part[warp * 64 + lane] = lo;
      part[warp * 64 + 32 + lane] = hi;
      __syncthreads();
      const int pc = threadIdx.x >> 6, h = (threadIdx.x >> 5) & 1;  // 64 threads finish one piece
      if (pc < kPieces && p0 + pc < npieces) {
        float4 o = part[pc * kSlices * 64 + h * 32 + lane];
#pragma unroll
        for (int sl = 1; sl < kSlices; ++sl) {
          const float4 a = part[(pc * kSlices + sl) * 64 + h * 32 + lane];
          o.x += a.x; o.y += a.y; o.z += a.z; o.w += a.w;
        }
        int m, n;
        grid.origin(p0 + pc, m, n);
        float4* out = place(m + lane, n + 4 * h);
        write(out, o, before(out));
      }
      __syncthreads();
    }
  }
}

// Shares of the sequences per piece: as many as still leave every warp resident at once (32 per SM) and eight sequences
// to sum per warp.  Past that a split only adds warps that wait their turn: 896 -> 896 at 16 sequences, two or more
// sequences per warp, took 18.9 us split against 12.5 us whole.
inline int combine_slices(long long npieces, int B, int sms) {
  int s = 1;
  while (s < 8 && npieces * 2 * s <= 32ll * sms && B >= 16 * s) s *= 2;
  return s;
}

// Sequences from which on a whole sum is a long one.  1536 -> 4096, long / short form: 15 sequences 46.7 / 33.4 us, 60: 113 /
// 111, 100: 177 / 181, 256: 463 / 467; 896 -> 4864: 15 sequences 36.1 / 25.2, 60: 83.2 / 77.5, 100: 125.9 / 124.5.
constexpr int kManySeqs = 64;

// Split store: dW = beta dW + sum_i (c_i / s_i) (hi_i + lo_i / 16).  One thread per PAIR of slots (two tile rows x 8
// columns), so that every load is 16 bytes per plane: with one slot per thread the two planes cost twice the load
// instructions per byte of the bf16 store and the pass fell to 5.0 TB/s inside the step.
// kDeep: registers for more of a thread's loads at once, on three CTAs per SM instead of four: where that takes no more waves.
// 200 sequences, 896 x 256 66 -> 40 us (four CTAs -> three), 896 x 896 77 -> 57, 2048 x 2048 (three waves instead of two) 249 -> 259.
template <bool kDeep>
__global__ void __launch_bounds__(256, kDeep ? 3 : 4) k_e4m3_combine(const uint2* __restrict__ planes, long long nchunks /* n_pad / 8 */,
                                                       int B, PieceGrid grid, int d_in, int d_out,
                                                       const float* __restrict__ coeffs, const float* __restrict__ scales,
                                                       float* __restrict__ dW, float beta,
                                                       const WsTag* __restrict__ tag_dev, WsTag tag,
                                                       int32_t* __restrict__ info) {
  pdl_wait();
  if (!ws_tag_matches(tag_dev, tag, info)) return;  // another layer's or microbatch's gradients: touch nothing
  __shared__ float sc[256];
  for (int i = threadIdx.x; i < B; i += blockDim.x) sc[i] = coeffs[i] / scales[i];
  __syncthreads();
  const long long npairs = nchunks / 2;
  for (long long pos = blockIdx.x * (long long)blockDim.x + threadIdx.x; pos < npairs;
       pos += (long long)gridDim.x * blockDim.x) {
    // pos = piece * 16 + pair of slots
    const int piece = (int)(pos >> 4), l = (int)(pos & 15) * 2;
    int m, n;
    grid.origin(piece, m, n);
    m += l;
    if (m >= d_out) continue;
    if (!ISOPO_IN_RANGE((long long)stored_slot((size_t)piece, B - 1, B, l + 1), nchunks * B, info, kIdCombine)) continue;
    if (!ISOPO_IN_RANGE((long long)m * d_in + n + 7, (long long)d_out * d_in, info, kIdCombine)) continue;
    float acc[16] = {};
    const uint4* hi = reinterpret_cast<const uint4*>(planes + stored_slot((size_t)piece, 0, B, l));
    const uint4* lo = reinterpret_cast<const uint4*>(planes + (size_t)nchunks * B + stored_slot((size_t)piece, 0, B, l));
    const size_t stride = 16;  // 16-byte units between successive sequences of one piece
    auto add = [&](const uint4& hv, const uint4& lv, float c) {
      const uint32_t hw[8] = {hv.x & 0xffffu, hv.x >> 16, hv.y & 0xffffu, hv.y >> 16,
                              hv.z & 0xffffu, hv.z >> 16, hv.w & 0xffffu, hv.w >> 16};
      const uint32_t lw[8] = {lv.x & 0xffffu, lv.x >> 16, lv.y & 0xffffu, lv.y >> 16,
                              lv.z & 0xffffu, lv.z >> 16, lv.w & 0xffffu, lv.w >> 16};
#pragma unroll
      for (int h = 0; h < 8; ++h) {
        // hi + lo / 16 in half precision is exact (4 + 4 significant bits, at most 9 binades apart)
        const float2 g = __half22float2(__hfma2(e4m3x2_to_half2(lw[h]), __float2half2_rn(1.f / kLoScale), e4m3x2_to_half2(hw[h])));
        acc[2 * h] = fmaf(c, g.x, acc[2 * h]);
        acc[2 * h + 1] = fmaf(c, g.y, acc[2 * h + 1]);
      }
    };
    constexpr int kN = kCombineInFlight / 2;
    int i = 0;
    for (; i + kN <= B; i += kN) {
      uint4 hv[kN], lv[kN];
#pragma unroll
      for (int u = 0; u < kN; ++u) { hv[u] = __ldcs(hi + (size_t)(i + u) * stride); lv[u] = __ldcs(lo + (size_t)(i + u) * stride); }
#pragma unroll
      for (int u = 0; u < kN; ++u) add(hv[u], lv[u], sc[i + u]);
    }
    for (; i < B; ++i) add(__ldcs(hi + (size_t)i * stride), __ldcs(lo + (size_t)i * stride), sc[i]);
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      if (m + r >= d_out) break;
      float4* out = reinterpret_cast<float4*>(dW + (size_t)(m + r) * d_in + n);
      float4 o0 = make_float4(acc[8 * r], acc[8 * r + 1], acc[8 * r + 2], acc[8 * r + 3]);
      float4 o1 = make_float4(acc[8 * r + 4], acc[8 * r + 5], acc[8 * r + 6], acc[8 * r + 7]);
      if (beta != 0.f) {
        const float4 p0 = out[0], p1 = out[1];
        o0.x += p0.x; o0.y += p0.y; o0.z += p0.z; o0.w += p0.w;
        o1.x += p1.x; o1.y += p1.y; o1.z += p1.z; o1.w += p1.w;
      }
      out[0] = o0;
      out[1] = o1;
    }
  }
}

}  // namespace

isopo_status plan_ntk(const WsLayout& L, int B, bool split, bool deterministic, NtkPlan* plan) {
  if (B > 256) return ISOPO_ERR_UNSUPPORTED;
  int dev = 0, sms = 0;
  ISOPO_CUDA_TRY(cudaGetDevice(&dev));
  ISOPO_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  // The least power of two that holds them, four at the least: rows of a box that do not exist are copied as slowly as any.  Boxes of 32
  // rows / as now: 888 x 3504, 4 sequences 18.7 / 8.9 us, whole call 7 sequences 40.7 / 32.3, 4752 x 96, 14 sequences 17.7 / 16.7.
  plan->box_rows = 256;
  while (plan->box_rows > 4 && plan->box_rows / 2 >= B) plan->box_rows /= 2;
  plan->ppb = 256 / plan->box_rows;
  // boxes along the contraction: four per piece group of bf16 (64 elements a row), two of e4m3 (128 elements a row)
  plan->nkb = (L.n_pad / kPieceElems + plan->ppb - 1) / plan->ppb * (split ? 2 : 4);
  // Four boxes of a CTA pay for its start, eight above 16 sequences: half of the CTAs are half of the additions to an entry of K (896 x 128,
  // 64 sequences: error 1.0e-7 with 56 of them, 1.4e-7 with 112, isopo_layer_gram 15.3 / 14.3 us; 512 x 512, 32: 1.2e-7 / 1.6e-7, 17.5 / 17.3).
  plan->grid = (int)std::max<long long>(1, std::min<long long>(sms, plan->nkb / (B > 16 ? 8 : 4)));
  if (deterministic) plan->grid = std::min(plan->grid, kNtkMaxPartials);
  // CTAs whose slab of the contraction is empty take no part
  const long long per = (plan->nkb + plan->grid - 1) / plan->grid;
  plan->n_active = (int)((plan->nkb + per - 1) / per);
  // K completed by the last CTA: a launch less (2 us for the host, which bounds a pass over little data: 128 x 128, 32
  // sequences 18.3 -> 16.1 us), but a CTA by itself is slower than a kernel that is set up when this one ends, the more so the
  // more sequences: 896 x 896, K and solve: 24.5 us both ways at 16, 31.5 / 30.4 at 32, 47.2 / 45.0 at 48, 127.6 / 117.1 at 128.
  plan->by_last = !deterministic && (B <= 16 || (B <= 32 && per <= 16));
  // Up to 32 sequences there are four groups of pieces or more in an accumulator, and two accumulators: their sums meet in shared memory
  // first.  Eight boxes of every CTA on the same 20 x 20 entries waited for one another: 4088 x 1440, 20 sequences 154 us by
  // atomics, 171 by boxes.
  plan->by_boxes = !deterministic && B > kNtkSmemSums && L.off_ksums != 0;
  return ISOPO_OK;
}

isopo_status bf16_ntk(const NtkPlan& plan, const void* G, const WsLayout& L, int B, float* K, float* acc, WsHead* head, float* kpart,
                      const StoreFmt& fmt, int32_t* info, cudaStream_t st) {
  if (fmt.split && kpart) return ISOPO_ERR_INVALID_ARG;  // the split store's diagonal is summed with float atomics
  CUtensorMap mapG, mapK;
  const uint32_t rows = (uint32_t)plan.box_rows, ppb = (uint32_t)plan.ppb;
  const uint64_t pieces = (uint64_t)(L.n_pad / kPieceElems);
  isopo_status s = fmt.split ? make_map_pieces_u8(&mapG, G, (uint64_t)B, pieces, rows, ppb)
                             : make_map_pieces_bf16(&mapG, G, (uint64_t)B, pieces, rows, ppb);
  if (s != ISOPO_OK) return s;
  if (plan.by_boxes) {
    if ((s = make_map_2d_f32(&mapK, acc, (uint64_t)B, (uint64_t)ntk_pitch(B), 32, false)) != ISOPO_OK) return s;
  } else {
    mapK = mapG;
  }
  auto kernel = plan.by_boxes ? (fmt.split ? k_bf16_ntk<true, kBoxes> : k_bf16_ntk<false, kBoxes>)
                : rows < 32   ? (fmt.split ? k_bf16_ntk<true, kFew> : k_bf16_ntk<false, kFew>)
                              : (fmt.split ? k_bf16_ntk<true, kRows> : k_bf16_ntk<false, kRows>);
  ISOPO_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes));
  NtkParams p{kpart, fmt.split ? fmt.scales : nullptr, K, B, plan.nkb, info, plan.box_rows, plan.ppb,
              plan.by_last ? &head->done : nullptr, (uint32_t)plan.n_active, fmt.kdiag};
  {
    LaunchScope scope(kIdNtk, st);
    launch(kernel, plan.grid, kThreads, kSmemBytes, st, mapG, mapK, p);
  }
  ISOPO_CUDA_TRY(cudaGetLastError());
  if (plan.by_last) return ISOPO_OK;
  {
    LaunchScope scope(kIdMirror, st);
    if (kpart) launch(k_ntk_reduce, (B * B + 255) / 256, 256, 0, st, kpart, plan.n_active, B, K);
    else launch(k_ntk_finish, (B * B + 255) / 256, 256, 0, st, acc, plan.by_boxes ? ntk_pitch(B) : B, K, B, fmt.split ? fmt.kdiag : nullptr);
  }
  ISOPO_CUDA_TRY(cudaGetLastError());
  return ISOPO_OK;
}

isopo_status mirror_upper(float* K, int B, cudaStream_t st) {
  {
    LaunchScope scope(kIdMirror, st);
    launch(k_mirror, (B * B + 255) / 256, 256, 0, st, K, B);
  }
  ISOPO_CUDA_TRY(cudaGetLastError());
  return ISOPO_OK;
}

isopo_status bf16_combine(const void* G, const WsLayout& L, int d_in, int d_out, int B, const float* coeffs, float* dW,
                          float beta, const WsTag* tag_dev, const WsTag& tag, const StoreFmt& fmt, int32_t* info,
                          cudaStream_t st) {
  if (B > 256) return ISOPO_ERR_UNSUPPORTED;
  const long long chunks = L.n_pad / 8;
  const PieceGrid pg = piece_grid(d_in, d_out);
  int dev = 0, sms = 0;
  ISOPO_CUDA_TRY(cudaGetDevice(&dev));
  ISOPO_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int slices = fmt.split ? 1 : combine_slices(chunks / 32, B, sms);
  const int grid = (int)std::min<long long>((chunks * slices + 255) / 256, (long long)sms * 8);
  {
    LaunchScope scope(kIdCombine, st);
    const int deep_waves = (grid + 3 * sms - 1) / (3 * sms), waves = (grid + 4 * sms - 1) / (4 * sms);
    if (fmt.split)
      launch(deep_waves <= waves ? k_e4m3_combine<true> : k_e4m3_combine<false>, grid, 256, 0, st, (const uint2*)G, chunks, B, pg,
             d_in, d_out, coeffs, fmt.scales, dW, beta, tag_dev, tag, info);
    else
      launch((slices == 1   ? (B >= kManySeqs ? k_bf16_combine<1, true> : k_bf16_combine<1, false>)
       : slices == 2 ? k_bf16_combine<2, false>
       : slices == 4 ? k_bf16_combine<4, false>
                     : k_bf16_combine<8, false>), grid, 256, 0, st, (const uint4*)G, chunks, B, pg, d_in, d_out, coeffs, dW, beta,
                                                                tag_dev, tag, info);
  }
  ISOPO_CUDA_TRY(cudaGetLastError());
  return ISOPO_OK;
}

}  // namespace isopo
