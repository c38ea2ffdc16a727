// sm_100a plumbing shared by the tensor-core kernels: mbarriers with bounded waits, TMA tile loads,
// tensor-memory allocation, tcgen05 MMA issue / commit / accumulator loads, descriptor builders.
// All inline PTX; no library templates.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "isopo_internal.h"

namespace isopo {
namespace tc {

// ---------------------------------------------------------------------------------------------
// Stored per-sequence gradients (bf16, materialised route; the order is private to the library).
//
// G_i is cut into "pieces" of 32 rows x 8 columns = 256 elements = 512 bytes: piece (tm, c, q) holds rows
// 128 tm + 32 q .. + 31 and columns 8 c .. 8 c + 7, row-major inside (row r at 16-byte slot r % 32).  That is exactly
// what one epilogue warp writes with one 16-byte store per lane.  Pieces are the OUTER index and
// the sequence the inner one:
//     uint4 index of (piece p, sequence i, slot l) = (p * B + i) * 32 + l
// so the B copies of one piece are contiguous (B x 512 bytes).  The NTK kernel contracts over
// pieces and reads each such block once, front to back; the combine kernel sums over i inside it.
// Any fixed order of the elements of G_i gives the same <G_i, G_j>.
// Within a 128-row tile the column groups follow one another, its row quarters innermost.  Only pieces that hold
// elements of G exist: d_in / 8 column groups and ceil(d_out / 32) row quarters, so a layer off the 128 x 256 tile
// grid stores and re-reads no padding columns (896 columns padded to 1024 were 14 % of the bytes of three passes).
// ---------------------------------------------------------------------------------------------
constexpr int kPieceElems = 256;
struct PieceGrid {
  int groups;    // column groups: d_in / 8
  int quarters;  // row quarters: ceil(d_out / 32)
  __host__ __device__ __forceinline__ int quarters_of(int tm) const {  // row quarters of 128-row tile tm (none past the end)
    const int left = quarters - 4 * tm;
    return left > 4 ? 4 : left;
  }
  __host__ __device__ __forceinline__ size_t piece(int tm, int c, int q) const {
    return (size_t)tm * 4 * (size_t)groups + (size_t)c * (size_t)quarters_of(tm) + (size_t)q;
  }
  // first row and first column of piece p
  __device__ __forceinline__ void origin(int p, int& m, int& n) const {
    const int per_tm = 4 * groups, tm = p / per_tm, rem = p - tm * per_tm, nq = quarters_of(tm);
    const int c = nq == 4 ? rem >> 2 : rem / nq;
    m = tm * kTileM + (rem - c * nq) * 32;
    n = c * 8;
  }
};
inline PieceGrid piece_grid(int d_in, int d_out) { return PieceGrid{d_in / 8, (d_out + 31) / 32}; }
__host__ __device__ __forceinline__ size_t stored_slot(size_t piece, int i, int B, int l) {
  return (piece * (size_t)B + (size_t)i) * 32 + (size_t)l;
}

// ---------------------------------------------------------------------------------------------
// host: tensor maps
// ---------------------------------------------------------------------------------------------

// Row-major bf16 matrix [rows, cols] viewed by TMA as (x = column, y = row); boxes of
// `box_cols` x `box_rows` elements land in shared memory with the 128-byte swizzle.
// box_cols * 2 bytes must be 128.  Out-of-range elements read as zero.
isopo_status make_map_2d_bf16(CUtensorMap* map, const void* base, uint64_t rows, uint64_t cols, uint64_t row_stride_elems,
                              uint32_t box_cols, uint32_t box_rows);

// Row-major float32 matrix [rows, cols], cols a multiple of 4, in boxes of 32 rows x `box_cols` (16 or 32: 64- or 128-byte swizzle):
// what a warp adds or writes.
isopo_status make_map_2d_f32(CUtensorMap* map, void* base, uint64_t rows, uint64_t cols, uint32_t box_cols, bool swizzle = true);

// Stored per-sequence gradients viewed as (x = element inside a 256-element piece row, y = sequence,
// z = piece): boxes of 64 elements x `box_rows` sequences x `box_pieces` pieces, 128-byte swizzle.  Sequences
// past B and pieces past the last read as zero.
isopo_status make_map_pieces_bf16(CUtensorMap* map, const void* base, uint64_t B, uint64_t pieces, uint32_t box_rows,
                                  uint32_t box_pieces);
// One e4m3 plane of the split store viewed as (x = byte inside a 256-byte piece row, y = sequence, z = piece): boxes of
// 128 bytes x `box_rows` sequences x `box_pieces` pieces, 128-byte swizzle.
isopo_status make_map_pieces_u8(CUtensorMap* map, const void* base, uint64_t B, uint64_t pieces, uint32_t box_rows,
                                uint32_t box_pieces);

// ---------------------------------------------------------------------------------------------
// device: generic helpers
// ---------------------------------------------------------------------------------------------

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ bool elect_one() {
  uint32_t pred;
  asm volatile(
      "{\n.reg .pred p;\nelect.sync _|p, 0xffffffff;\nselp.u32 %0, 1, 0, p;\n}\n" : "=r"(pred));
  return pred != 0;
}

// ---- mbarrier ----
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void fence_barrier_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

// One look at the barrier, never blocks.
__device__ __forceinline__ bool mbar_test_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n.reg .pred p;\nmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

// Bounded wait.  Gives up after `limit` clock ticks (by default ~2^31, about a second) or as soon as
// another role of this CTA has given up (`*abort_flag` != 0, shared memory); records
// ISOPO_INFO_TIMEOUT | code in *info (only over a zero) and returns false.  Callers leave their loops
// and fall through to the common teardown, so the kernel always ends and the context stays usable.
constexpr long long kWaitLimitClocks = 1ll << 31;
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, int32_t* info,
                                          int code, long long limit = kWaitLimitClocks) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long start = clock64();
  while (true) {
    for (int i = 0; i < 64; ++i)
      if (mbar_try_wait(bar, parity)) return true;
    if (*abort_flag) return false;
    if (clock64() - start > limit) {
      *abort_flag = 1;
      atomicCAS(info, 0, ISOPO_INFO_TIMEOUT | code);
      return false;
    }
  }
}

// ---- TMA ----
__device__ __forceinline__ void prefetch_tensormap(const CUtensorMap* m) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(m)) : "memory");
}
// x = innermost (column) coordinate, a multiple of 8 bf16 elements (16 bytes); y = row.
__device__ __forceinline__ void tma_load_2d(uint32_t dst_smem, const CUtensorMap* map, int x, int y, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
      ::"r"(dst_smem), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst_smem, const CUtensorMap* map, int x, int y, int z, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
      ::"r"(dst_smem), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(bar)
      : "memory");
}
// As tma_load_2d inside a CTA pair: the barrier may live in the other CTA of the pair (`bar` is a
// shared::cluster address); the data still lands in this CTA.  No multicast.
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst_smem, const CUtensorMap* map, int x, int y, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
      ::"r"(dst_smem), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
      : "memory");
}
// A box from shared memory to where it stands in global memory, written or added; what lies outside the matrix is left out.
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, int x, int y, uint32_t src_smem) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];"
               ::"l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(src_smem)
               : "memory");
}
__device__ __forceinline__ void tma_add_2d(const CUtensorMap* map, int x, int y, uint32_t src_smem) {
  asm volatile("cp.reduce.async.bulk.tensor.2d.global.shared::cta.add.bulk_group [%0, {%1, %2}], [%3];"
               ::"l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(src_smem)
               : "memory");
}
// Lane's row of a 32-row box in shared memory (`box`, a multiple of 1024 bytes), its 16-byte groups where the tensor map's swizzle
// has them; no bank conflicts.
__device__ __forceinline__ void box_row(uint32_t box, int lane, const uint32_t (&r)[32]) {
#pragma unroll
  for (int v = 0; v < 8; ++v)
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(box + lane * 128 + ((v ^ (lane & 7)) << 4)), "r"(r[4 * v]),
                 "r"(r[4 * v + 1]), "r"(r[4 * v + 2]), "r"(r[4 * v + 3]) : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
template <int kPending>
__device__ __forceinline__ void bulk_wait_read() {  // all but the last kPending groups of this thread have read their source (what they write is complete when the kernel is)
  asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(kPending) : "memory");
}
// generic-proxy writes to shared memory -> visible to the async proxy (TMA, tcgen05.mma)
__device__ __forceinline__ void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// ---- tensor memory ----
__device__ __forceinline__ void tmem_alloc(uint32_t slot_smem, uint32_t ncols) {  // one full warp
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot_smem), "r"(ncols) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {  // one full warp
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// D[tmem] (+)= A[smem] * B[smem], bf16 inputs, float32 accumulate; issued by ONE thread.
__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                         bool accumulate) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"((uint32_t)accumulate)
      : "memory");
}
// The same with e4m3 A and B (kind::f8f6f4: 32 elements of the contraction per instruction, float32 accumulate).
__device__ __forceinline__ void mma_e4m3(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                         bool accumulate) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n}\n"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"((uint32_t)accumulate)
      : "memory");
}
// Arrives on `bar` once every MMA issued so far by this thread has completed.
__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// 32 consecutive float32 columns of this warp's 32 accumulator rows (lane l reads row l of the
// warp's quarter).  taddr = (first lane << 16) | first column.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// ---- CTA pairs (cluster of two CTAs driving one 2-CTA tcgen05.mma) ----
__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// shared::cluster address of the same shared-memory location in CTA `rank` of this cluster
__device__ __forceinline__ uint32_t map_to_cta(uint32_t smem_addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {  // every thread of both CTAs
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Arrival on a barrier of the other CTA of the pair (CTA-scope release: it says "done", it is not a
// cluster-wide fence, which would stall the arriving warp for hundreds of clocks).
__device__ __forceinline__ void mbar_arrive_remote(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
__device__ __forceinline__ void st_cluster_u32(uint32_t cluster_addr, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(cluster_addr), "r"(v) : "memory");
}
// Bounded wait inside a CTA pair: as mbar_wait, and on giving up it also raises the peer's abort
// flag (`peer_abort`, a shared::cluster address) so that both CTAs of the pair head for the teardown.
__device__ __forceinline__ bool mbar_wait_pair(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                               uint32_t peer_abort, int32_t* info, int code) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long start = clock64();
  while (true) {
    for (int i = 0; i < 64; ++i)
      if (mbar_try_wait(bar, parity)) return true;
    if (*abort_flag) return false;
    if (clock64() - start > kWaitLimitClocks) {
      *abort_flag = 1;
      st_cluster_u32(peer_abort, 1u);
      atomicCAS(info, 0, ISOPO_INFO_TIMEOUT | code);
      return false;
    }
  }
}
__device__ __forceinline__ void tmem_alloc_pair(uint32_t slot_smem, uint32_t ncols) {  // one full warp in EACH CTA
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot_smem), "r"(ncols) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {  // one full warp in EACH CTA
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
// 2-CTA MMA, issued by ONE thread of the pair's first CTA: each CTA supplies its half of A's rows
// and of B's rows (same shared-memory offsets in both) and receives its half of D's rows.
__device__ __forceinline__ void mma_bf16_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                              bool accumulate) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"((uint32_t)accumulate)
      : "memory");
}
// Arrives on the barrier at this shared-memory offset in BOTH CTAs of the pair once every MMA
// issued so far by this thread has completed.
__device__ __forceinline__ void mma_commit_pair(uint32_t bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
      ::"r"(bar), "h"((uint16_t)3)
      : "memory");
}

// ---- descriptors ----
// Instruction descriptor, kind::f16 with bf16 A and B, float32 D.  a_mn / b_mn: operand is stored
// with its M (resp. N) index contiguous ("MN-major") instead of its K index.
__host__ __device__ constexpr uint32_t make_idesc_bf16(int M, int N, bool a_mn, bool b_mn) {
  return (1u << 4)                       // D format: float32
         | (1u << 7) | (1u << 10)        // A, B format: bf16
         | ((a_mn ? 1u : 0u) << 15) | ((b_mn ? 1u : 0u) << 16)
         | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// Instruction descriptor, kind::f8f6f4 with e4m3 A and B (format code 0), float32 D, both operands K-major.
__host__ __device__ constexpr uint32_t make_idesc_e4m3(int M, int N) {
  return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// Shared-memory matrix descriptor for 128-byte-swizzled tiles (rows of 128 bytes, 8-row groups of
// 1024 bytes, tile base 1024-byte aligned).
//   K-major operand  (row = M/N index, 64 bf16 of K per row): sbo = bytes between 8-row groups.
//   MN-major operand (row = K index, 64 bf16 of M/N per row): sbo = bytes between 8-row K groups,
//                    lbo = bytes between successive 64-element chunks of M/N.
__device__ __forceinline__ uint64_t make_sdesc_sw128(uint32_t smem_addr, uint32_t lbo_bytes, uint32_t sbo_bytes) {
  return (uint64_t)((smem_addr & 0x3FFFFu) >> 4) | ((uint64_t)(lbo_bytes >> 4) << 16) |
         ((uint64_t)(sbo_bytes >> 4) << 32) | (1ull << 46) | (2ull << 61);
}

// K[j][i] = K[i][j] for the pairs of which one triangle is filled (kFromUpper: i < j), and the diagonal where `set_diag`, by
// the 128 threads r = 0 .. 127 of one CTA once every CTA's additions are visible.  Reads run along rows; the scattered
// writes need not be waited for.
template <bool kFromUpper, typename Diag>
__device__ __forceinline__ void mirror_by_cta(float* K, int B, int r, Diag diag, bool set_diag) {
  const int total = B * B;
  for (int e0 = r; e0 < total; e0 += 128 * 8) {
    float v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = e0 + u * 128 < total ? __ldcg(K + e0 + u * 128) : 0.f;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int e = e0 + u * 128, i = e / B, j = e - i * B;
      if (e < total && (kFromUpper ? j > i : j < i)) K[(size_t)j * B + i] = v[u];
      else if (set_diag && e < total && j == i) K[e] = diag(i);
    }
  }
}

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);  // .x = lo (low 16 bits)
  return *reinterpret_cast<uint32_t*>(&v);
}

// two floats -> two e4m3 bytes (`a` in the low byte), round to nearest even, saturating at +-448
__device__ __forceinline__ uint32_t pack_e4m3x2(float a, float b) {
  uint16_t r;
  asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(r) : "f"(b), "f"(a));
  return r;
}
// two e4m3 bytes -> two halves / two floats (exact)
__device__ __forceinline__ __half2 e4m3x2_to_half2(uint32_t v) {
  uint32_t h2;
  asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(h2) : "h"((uint16_t)v));
  return *reinterpret_cast<__half2*>(&h2);
}
__device__ __forceinline__ float2 unpack_e4m3x2(uint32_t v) { return __half22float2(e4m3x2_to_half2(v)); }
constexpr float kLoScale = 16.f;  // the `lo` plane of the split store holds 16 x the residual of the `hi` plane

}  // namespace tc
}  // namespace isopo
