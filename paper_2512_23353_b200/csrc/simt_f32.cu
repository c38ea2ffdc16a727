// float32 kernels of the ISOPO layer path (parity to 1e-5), plus the token -> sequence map that both
// dtypes use.  Token contractions are float32 FMA; everything that sums over many products of
// products (K) is accumulated in float64.
#include <algorithm>
#include <atomic>

#include "isopo_internal.h"
#include "slab_plan.h"

namespace isopo {

namespace {

// Host values travel to the device as kernel arguments: no hidden synchronisation with the stream, and nothing that reads
// the caller's array after the call returns.
constexpr int64_t kSms = 148;  // of a B200: the rules below that fill the machine
template <int kN>
__global__ void __launch_bounds__(256) k_store_offsets(const __grid_constant__ OffsetArgs<kN> a, int64_t base, int n,
                                                       int64_t* __restrict__ off) {
  pdl_wait();
  const int32_t* from = offsets_memory(a);
  for (int t = threadIdx.x; t < n; t += blockDim.x) off[base + t] = from[t];
}

// What a kernel over all tokens needs before it starts, in one launch: the offsets in the workspace, the regions it adds
// into cleared, and per token its sequence (kOut = kTokSeq) or that sequence's coefficient (kTokScale).
enum PrepOut { kOffsetsOnly, kTokSeq, kTokScale };
template <int kOut, typename Off>
__device__ __forceinline__ void fill_tokens(const Off* off, int B, int64_t T, const float* __restrict__ coeffs, void* __restrict__ out) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < T; t += (int64_t)gridDim.x * blockDim.x) {
    int lo = 0, hi = B;  // invariant: off[lo] <= t < off[hi]
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (off[mid] <= (Off)t) lo = mid; else hi = mid;
    }
    if (kOut == kTokScale) static_cast<float*>(out)[t] = coeffs[lo];
    else static_cast<int32_t*>(out)[t] = lo;
  }
}
// offsets in the arguments: every CTA copies them to shared memory and searches there; CTA 0 also leaves them in the workspace
template <int kOut, int kN>
__global__ void __launch_bounds__(256) k_prep(const __grid_constant__ OffsetArgs<kN> a, int B, int64_t T,
                                              int64_t* __restrict__ off_dev, const float* __restrict__ coeffs,
                                              void* __restrict__ out, const __grid_constant__ Clear clear) {
  __shared__ int32_t s_off[kN];
  const int32_t* from = offsets_memory(a);
  for (int i = threadIdx.x; i <= B; i += blockDim.x) s_off[i] = from[i];
  pdl_wait();
  __syncthreads();
  if (blockIdx.x == 0)
    for (int i = threadIdx.x; i <= B; i += blockDim.x) off_dev[i] = s_off[i];
  clear_regions(clear);
  if (kOut != kOffsetsOnly) fill_tokens<kOut>(s_off, B, T, coeffs, out);
}
// k_prep<kTokSeq>, and rows copied to a pitch of whole lines, a warp to a row.  HBM stream: 40,000 tokens, 3064 + 712 columns 112 us.
template <int kN>
__global__ void __launch_bounds__(256) k_prep_repitch(const __grid_constant__ OffsetArgs<kN> a, int B, int64_t T,
                                                      int64_t* __restrict__ off_dev, int32_t* __restrict__ out,
                                                      const __grid_constant__ Clear clear, const __grid_constant__ Repitch rp) {
  __shared__ int32_t s_off[kN];
  const int32_t* from = offsets_memory(a);
  for (int i = threadIdx.x; i <= B; i += blockDim.x) s_off[i] = from[i];
  pdl_wait();
  __syncthreads();
  if (blockIdx.x == 0)
    for (int i = threadIdx.x; i <= B; i += blockDim.x) off_dev[i] = s_off[i];
  clear_regions(clear);
  fill_tokens<kTokSeq>(s_off, B, T, nullptr, out);
  const int lane = threadIdx.x & 31, warps = gridDim.x * (blockDim.x >> 5);
#pragma unroll
  for (int o = 0; o < kMaxRepitch; ++o) {
    if (o >= rp.n) break;
    const int d8 = rp.d8[o];
    for (int64_t t = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); t < T; t += warps) {
      const uint4* src = rp.src[o] + t * d8;
      uint4* dst = rp.dst[o] + t * rp.p8[o];
      for (int e0 = lane; e0 < d8; e0 += 128) {
        uint4 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (e0 + 32 * u < d8) v[u] = __ldcs(src + e0 + 32 * u);
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (e0 + 32 * u < d8) dst[e0 + 32 * u] = v[u];
      }
    }
  }
}
// more sequences than the arguments hold: k_store_offsets has left the offsets in the workspace
template <int kOut>
__global__ void __launch_bounds__(256) k_prep_many(const int64_t* __restrict__ off_dev, int B, int64_t T,
                                                   const float* __restrict__ coeffs, void* __restrict__ out,
                                                   const __grid_constant__ Clear clear) {
  pdl_wait();
  clear_regions(clear);
  if (kOut != kOffsetsOnly) fill_tokens<kOut>(off_dev, B, T, coeffs, out);
}

// ---------------------------------------------------------------------------------------------
// Register-blocked float32 GEMM over tokens: acc[p][q] += w_t * dY[t, m] * X[t, n] for tokens [t0, t1), tile
// kTile x kTile, kT x kT elements per thread.  Token rows are staged kTK at a time by cp.async, kStages deep (16-byte
// copies where the row length allows, 4-byte ones otherwise; columns and tokens past the end arrive as zeros); a thread's
// rows and columns come in groups of four, so that its operands are 16-byte shared loads.  Two neighbouring columns share
// one packed fma (fma.rn.f32x2: the same two roundings, half the issue slots, which the shared loads need).
// Bound by the float32 pipe: 64 sequences of 72 tokens, 896 x 896: 174 us (42 TFLOP/s with the 205 MB store of G) against
// 342 us with a 64 x 64 tile loaded synchronously.  Stages of 8 tokens waste less of a short sequence's last stage
// (G_i: 174 against 187 us with 16); over one long token range stages of 16 synchronise half as often (dW: 197 against 212 us).
// The copies' addresses are stepped, not computed per element, and a token's weight is copied like its row: dW of 4835 tokens
// 190 -> 177 us, 895 x 895 (4-byte copies) 230 -> 199, G of 64 sequences of 75 tokens, 895 x 895, 285 -> 234.
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ void cp_async16(void* dst, const void* src, bool live) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src),
               "r"(live ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async4(void* dst, const void* src, bool live) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src),
               "r"(live ? 4 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int kPending>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(kPending) : "memory"); }

typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// Stages rows [t, t + kRows) x columns [c0, c0 + kCols) of a row-major [., d] matrix into dst[kRows][kCols].  A thread keeps its
// column (group) and steps through the rows by address.
template <int kRows, int kCols, int kThreadsF>
__device__ __forceinline__ void stage_rows(float* dst, const float* __restrict__ M, int64_t t, int64_t t_end, int c0, int d) {
  const int left = (int)min((int64_t)kRows, t_end - t);  // rows that exist
  if ((d & 3) == 0) {
    constexpr int kStep = kThreadsF / (kCols / 4);
    const int r = threadIdx.x / (kCols / 4), c = threadIdx.x % (kCols / 4) * 4;
    if (kStep > kRows && r >= kRows) return;
    const bool col = c0 + c < d;
    const float* src = M + (t + r) * d + c0 + c;
    float* to = dst + r * kCols + c;
#pragma unroll
    for (int i = 0; i < kRows; i += kStep, src += (int64_t)kStep * d) {
      const bool live = col && r + i < left;
      cp_async16(to + i * kCols, live ? src : M, live);
    }
  } else {
    constexpr int kStep = kThreadsF / kCols;
    const int r = threadIdx.x / kCols, c = threadIdx.x % kCols;
    const bool col = c0 + c < d;
    const float* src = M + (t + r) * d + c0 + c;
    float* to = dst + r * kCols + c;
#pragma unroll
    for (int i = 0; i < kRows; i += kStep, src += (int64_t)kStep * d) {
      const bool live = col && r + i < left;
      cp_async4(to + i * kCols, live ? src : M, live);
    }
  }
}

template <int kTile, int kT, int kTK, int kStages>
struct TokenGemm {
  static constexpr int kSide = kTile / kT;                        // threads along one side
  static constexpr int kThr = kSide * kSide;
  static constexpr int kStage = kTK * 2 * kTile;                  // floats
  static constexpr int kSmem = kStages * (kStage + kTK) * 4;      // bytes (the last kTK floats: token weights)
  static_assert(kSmem <= 99 * 1024, "two CTAs per SM");
  f32x2 acc[kT][kT / 2];
  // tile row of acc[p][.], tile column of the first element of a pair acc[.][q / 2]
  __device__ __forceinline__ static int row(int p, unsigned tid) { return (p / 4) * (kTile / (kT / 4)) + (int)(tid / kSide) * 4 + p % 4; }
  __device__ __forceinline__ static int row(int p) { return row(p, threadIdx.x); }
  __device__ __forceinline__ static int col(int q, unsigned tid) { return (q / 4) * (kTile / (kT / 4)) + (int)(tid % kSide) * 4 + q % 4; }
  __device__ __forceinline__ static int col(int q) { return col(q, threadIdx.x); }

  // kScaled: the dY row of token t counts tokscale[t] times (rounded once, as a scaled copy of dY would be)
  template <bool kScaled>
  __device__ __forceinline__ void run(float* smem, const float* __restrict__ X, const float* __restrict__ dY, int d_in,
                                      int d_out, int64_t t0, int64_t t1, int m0, int n0, const float* __restrict__ tokscale) {
#pragma unroll
    for (int p = 0; p < kT; ++p)
#pragma unroll
      for (int q = 0; q < kT / 2; ++q) acc[p][q] = 0ull;
    const int nk = (int)((t1 - t0 + kTK - 1) / kTK);
    float* sw = smem + kStages * kStage;
    auto fetch = [&](int k) {
      if (k < nk) {
        float* s = smem + (k % kStages) * kStage;
        const int64_t t = t0 + (int64_t)k * kTK;
        stage_rows<kTK, kTile, kThr>(s, dY, t, t1, m0, d_out);
        stage_rows<kTK, kTile, kThr>(s + kTK * kTile, X, t, t1, n0, d_in);
        if (kScaled && threadIdx.x < kTK) {
          const bool live = t + threadIdx.x < t1;
          cp_async4(sw + (k % kStages) * kTK + threadIdx.x, live ? tokscale + t + threadIdx.x : tokscale, live);
        }
      }
      cp_async_commit();
    };
#pragma unroll
    for (int k = 0; k < kStages - 1; ++k) fetch(k);
    for (int k = 0; k < nk; ++k) {
      cp_async_wait<kStages - 2>();
      __syncthreads();  // stage k is complete for everybody, and everybody is done with the stage fetched next
      fetch(k + kStages - 1);
      const float* sY = smem + (k % kStages) * kStage;
      const float* sX = sY + kTK * kTile;
#pragma unroll
      for (int r = 0; r < kTK; ++r) {
        float a[kT];
        f32x2 b[kT / 2];
#pragma unroll
        for (int p = 0; p < kT; p += 4) {
          const float4 v = *reinterpret_cast<const float4*>(sY + r * kTile + row(p));
          a[p] = v.x; a[p + 1] = v.y; a[p + 2] = v.z; a[p + 3] = v.w;
        }
        if (kScaled) {
          const float w = sw[(k % kStages) * kTK + r];
#pragma unroll
          for (int p = 0; p < kT; ++p) a[p] *= w;
        }
#pragma unroll
        for (int q = 0; q < kT; q += 4) {
          const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(sX + r * kTile + col(q));
          b[q / 2] = v.x; b[q / 2 + 1] = v.y;
        }
#pragma unroll
        for (int p = 0; p < kT; ++p) {
          const f32x2 ap = pack2(a[p], a[p]);
#pragma unroll
          for (int q = 0; q < kT / 2; ++q) acc[p][q] = fma2(ap, b[q], acc[p][q]);
        }
      }
    }
  }
};
template <int kTile, int kT> using SeqGemm = TokenGemm<kTile, kT, 8, 4>;
template <int kTile, int kT> using SlabGemm = TokenGemm<kTile, kT, 16, 3>;

// G_i = dY_i^T X_i, one (tile, sequence) per CTA.  The launch also leaves the workspace tag and clears the K pass's count of
// finished CTAs.  Offsets come as kernel arguments when they fit (kArgOff), else from `off`.
struct F32StoredArgs {
  const float* X;
  const float* dY;
  int d_in, d_out, B;
  int64_t gstride;   // floats between the gradients of two sequences (a multiple of 4)
  const int64_t* off;
  float* G;
  uint32_t* done;    // CTAs of the K pass that have finished
  WsTag tag;
  WsTag* tag_dev;
};
template <bool kArgOff> struct OffsetParam { int64_t v[1]; };
template <> struct OffsetParam<true> { int32_t v[kArgChunk]; };
static_assert(sizeof(F32StoredArgs) + sizeof(OffsetParam<true>) <= 4096, "kernel arguments");

template <int kTile, int kT, bool kArgOff>
__global__ void __launch_bounds__(SeqGemm<kTile, kT>::kThr, kT == 8 ? 2 : 3)  // 64-wide: three CTAs 297 x 651, 55 x 256 tokens 279 -> 252 us
k_f32_seq_grad(const __grid_constant__ F32StoredArgs a, const __grid_constant__ OffsetParam<kArgOff> o) {
  pdl_wait();
  extern __shared__ __align__(16) float smem[];
  const int i = blockIdx.z, m0 = blockIdx.y * kTile, n0 = blockIdx.x * kTile;
  const int64_t cta = ((int64_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
  if (cta == 0) {
    if (threadIdx.x < 8) a.tag_dev->v[threadIdx.x] = a.tag.v[threadIdx.x];
    if (threadIdx.x == 8) *a.done = 0u;
  }
  const int64_t t0 = kArgOff ? o.v[i] : a.off[i], t1 = kArgOff ? o.v[i + 1] : a.off[i + 1];
  SeqGemm<kTile, kT> g;
  g.template run<false>(smem, a.X, a.dY, a.d_in, a.d_out, t0, t1, m0, n0, nullptr);
  float* Gi = a.G + (size_t)i * a.gstride;
#pragma unroll
  for (int p = 0; p < kT; ++p) {
    const int m = m0 + g.row(p);
    if (m >= a.d_out) continue;
#pragma unroll
    for (int q = 0; q < kT; q += 4) {
      const int n = n0 + g.col(q);
      float4 v;
      unpack2(g.acc[p][q / 2], v.x, v.y);
      unpack2(g.acc[p][q / 2 + 1], v.z, v.w);
      float* dst = Gi + (size_t)m * a.d_in + n;
      if ((a.d_in & 3) == 0) {
        if (n < a.d_in) *reinterpret_cast<float4*>(dst) = v;
      } else {
        if (n < a.d_in) dst[0] = v.x;
        if (n + 1 < a.d_in) dst[1] = v.y;
        if (n + 2 < a.d_in) dst[2] = v.z;
        if (n + 3 < a.d_in) dst[3] = v.w;
      }
    }
  }
  // the K pass reads whole groups of four: the padding of a gradient is zero
  if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x < 4) {
    const int64_t e = (int64_t)a.d_in * a.d_out + threadIdx.x;
    if (e < a.gstride) Gi[e] = 0.f;
  }
}

// dW += (c_seq(t) dY)^T X over a slab of tokens (split over blockIdx.z), float atomics; one slab that nothing is added to (`store`) is
// written.  The sums go through shared memory, so that a warp's additions are of whole lines of dW.
template <int kTile, int kT>
__global__ void __launch_bounds__(SlabGemm<kTile, kT>::kThr, kT == 8 ? 2 : 1)
k_f32_weight_grad(const float* __restrict__ X, const float* __restrict__ dY, int64_t T, int d_in, int d_out,
                  const float* __restrict__ tokscale, float* __restrict__ dW, int64_t slab, bool store) {
  pdl_wait();
  extern __shared__ __align__(16) float smem[];
  typedef SlabGemm<kTile, kT> Gemm;
  const int64_t t0 = blockIdx.z * slab, t1 = min(T, t0 + slab);
  Gemm g;
  g.template run<true>(smem, X, dY, d_in, d_out, t0, t1, blockIdx.y * kTile, blockIdx.x * kTile, tokscale);
  constexpr int kPass = kTile / (kT / 4), kPitch = kTile + 4;  // rows that four of a thread's p make up
  static_assert(kPass * kPitch * 4 <= Gemm::kSmem, "the sums reuse the stages");
  // 128 x 128: read anew, as keeping them through the GEMM takes registers that are not there (40 bytes of spills for 12: 7032 tokens, 1481 x
  // 1513 830 -> 768 us)
  unsigned tid = threadIdx.x, bx = blockIdx.x, by = blockIdx.y;
  if (kTile == 128) asm volatile("mov.u32 %0, %%tid.x;\nmov.u32 %1, %%ctaid.x;\nmov.u32 %2, %%ctaid.y;" : "=r"(tid), "=r"(bx), "=r"(by));
  const int m0 = by * kTile, n0 = bx * kTile;
  const bool quads = (d_in & 3) == 0 && (reinterpret_cast<uintptr_t>(dW) & 15) == 0;
#pragma unroll
  for (int p0 = 0; p0 < kT; p0 += 4) {
    __syncthreads();
#pragma unroll
    for (int p = p0; p < p0 + 4; ++p)
#pragma unroll
      for (int q = 0; q < kT; q += 4) {
        float4 v;
        unpack2(g.acc[p][q / 2], v.x, v.y);
        unpack2(g.acc[p][q / 2 + 1], v.z, v.w);
        *reinterpret_cast<float4*>(smem + (Gemm::row(p, tid) - p0 / 4 * kPass) * kPitch + Gemm::col(q, tid)) = v;
      }
    __syncthreads();
    const int first = m0 + p0 / 4 * kPass, rows = min(kPass, d_out - first);
    if (quads) {
      constexpr int kLanes = kTile / 4;
      const int c = tid % kLanes * 4;
      if (n0 + c < d_in)
#pragma unroll 1
        for (int r = tid / kLanes; r < rows; r += Gemm::kThr / kLanes) {
          const float4 v = *reinterpret_cast<const float4*>(smem + r * kPitch + c);
          float* at = dW + (size_t)(first + r) * d_in + n0 + c;
          if (store) *reinterpret_cast<float4*>(at) = v;
          else asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(at), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
        }
    } else {
      const int c = tid % kTile;
      if (n0 + c < d_in)
#pragma unroll 1
        for (int r = tid / kTile; r < rows; r += Gemm::kThr / kTile) {
          float* at = dW + (size_t)(first + r) * d_in + n0 + c;
          if (store) *at = smem[r * kPitch + c];
          else atomicAdd(at, smem[r * kPitch + c]);
        }
    }
  }
}

// ---------------------------------------------------------------------------------------------
// K_ij = sum(G_i * G_j), i <= j, products and sums in float64 (mma.sync m16n8k8.f64: the exact product of two floats,
// accumulated in float64).  A CTA takes every gridDim.y-th 64-column chunk of a pair of row blocks of G_flat, staged by
// cp.async as floats; its four warps share the columns of a chunk, each holding the whole block of K in registers, so a
// fragment is read and widened once for many MMAs.  kDiag: 8 kNB rows against themselves, only the 16 x 8 blocks on and
// above the diagonal; otherwise 16 kMA rows against 8 kNB others.  Every CTA stores its sums, and they are added in the order
// of the chunks (k_f32_ntk_finish, or the last CTA to finish where there are few): K is the same to the bit from run to run,
// which float64 atomics would not leave it where products cancel.  G and K, atomics / this: 64 sequences of 896 x 896 210 / 193
// us, 64 of 64 x 64 32.8 / 22.5, 16 of 896 x 896 64.8 / 40.5, 256 of 512 x 512 973 / 939, 3 of 896 x 896 24.9 / 26.6.
// Bound by the float64 pipe.  One CTA per pair (i, j) with scalar float64 additions re-read G B / 2 times: 1384 us at 64
// sequences of an 896 x 896 layer against 146 us, 3694 against 500 us at 256 sequences of 300 x 500.  One CTA of eight
// warps per SM instead of two of four: 162 and 715 us.  Few sequences leave the pass to HBM and need more loads in flight: kGroups.
// ---------------------------------------------------------------------------------------------
constexpr int kNtkKC = 64;             // columns per chunk
constexpr int kNtkPitch = kNtkKC + 4;  // floats: the 32 lanes of a fragment read hit 32 banks
constexpr int kNtkStages = 3;
constexpr int kNtkRows = 64;           // sequences per row block
constexpr int kNtkThreads = 128;

__device__ __forceinline__ void dmma16x8x8(double (&c)[4], double a0, double a1, double a2, double a3, double b0, double b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k8.row.col.f64.f64.f64.f64 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+d"(c[0]), "+d"(c[1]), "+d"(c[2]), "+d"(c[3])
      : "d"(a0), "d"(a1), "d"(a2), "d"(a3), "d"(b0), "d"(b1));
}

// 16 x 8 blocks of K in a warp's registers
constexpr int ntk_blocks(int ma, int nb, bool diag) { return diag ? ma * (ma + 1) : ma * nb; }
// The sums of one K pass: pairs x slabs CTAs, `doubles` of each, element (blk * 4 + q) * 32 + lane as the registers have them.
struct NtkParts {
  int64_t pairs, slabs;
  int ma, nb, doubles, groups;
  bool diag;
  __host__ __device__ int64_t total() const { return pairs * slabs * doubles; }
};
// First row of the row blocks of a pair: diagonal blocks in order; otherwise pairs I < J of 64-row blocks, I in two halves of
// 32 rows.
__device__ __forceinline__ void ntk_pair_rows(bool diag, int64_t pair, int& i0, int& j0) {
  if (diag) {
    i0 = j0 = (int)pair * kNtkRows;
    return;
  }
  int J = 1, r = (int)(pair >> 1);
  while (r >= J) { r -= J; ++J; }
  i0 = r * kNtkRows + (int)(pair & 1) * 32;
  j0 = J * kNtkRows;
}
// Adds shares first .. last - 1 of an element in order, kFlight loads in flight.
template <int kFlight>
__device__ __forceinline__ double ntk_sum(const double* part, int64_t stride, int first, int last) {
  double s = 0.0;
  for (int k = first; k < last; k += kFlight) {
    double v[kFlight];
#pragma unroll
    for (int u = 0; u < kFlight; ++u) v[u] = k + u < last ? __ldcg(part + (k + u) * stride) : 0.0;
#pragma unroll
    for (int u = 0; u < kFlight; ++u) s += v[u];
  }
  return s;
}
// Row and column of K that element e of a pair's block stands for; false where it is not of use.
__device__ __forceinline__ bool ntk_entry(const NtkParts& P, int i0, int j0, int e, int B, int& i, int& j) {
  const int lane = e & 31, q = (e >> 5) & 3;
  int p = 0, n = e >> 7;
  if (P.diag) {
    while (n >= P.nb - 2 * p) { n -= P.nb - 2 * p; ++p; }
    n += 2 * p;
  } else {
    p = n / P.nb;
    n -= p * P.nb;
  }
  i = i0 + p * 16 + (lane >> 2) + (q >> 1) * 8;
  j = j0 + n * 8 + 2 * (lane & 3) + (q & 1);
  return i <= j && j < B;
}
// Entry e of the upper triangle of B rows (by rows), and the element of the first diagonal block that stands for it.
__device__ __forceinline__ int ntk_triangle(const NtkParts& P, int B, int e, int& i, int& j) {
  i = 0;
  while (i < B && e >= B - i) { e -= B - i; ++i; }
  j = i + e;
  const int p = i >> 4, n = j >> 3, blk = p * (P.nb - p + 1) + n - 2 * p;
  return (blk * 4 + ((i >> 3) & 1) * 2 + (j & 1)) * 32 + (i & 7) * 4 + ((j & 7) >> 1);
}
__device__ __forceinline__ void ntk_write(float* __restrict__ K, int B, int i, int j, double v) {
  K[(size_t)i * B + j] = (float)v;
  K[(size_t)j * B + i] = (float)v;
}

template <int kMA, int kNB, bool kDiag, int kG>
struct NtkShape {
  static constexpr int kRowsStaged = kDiag ? 8 * kNB : 16 * kMA + 8 * kNB;
  static constexpr int kStageFloats = kRowsStaged * kNtkPitch;
  static constexpr int kSmemStages = kNtkStages * kStageFloats * 4;
  static constexpr int kBlocks = ntk_blocks(kMA, kNB, kDiag);
  static constexpr int kSmemRed = 2 * kBlocks * 128 * 8;               // two warps' blocks
  static constexpr int kSmemGroup = kSmemStages > kSmemRed ? kSmemStages : kSmemRed;
  // Few sequences leave the pass to HBM: kG groups of four warps, each with a ring and chunks of its own, share a CTA, so that
  // their sums meet in shared memory and there are few shares of K to add.  Small layers spread the groups over the SMs instead.
  static constexpr int kGroups = kG;
  static constexpr int kThr = kGroups * kNtkThreads;
  static constexpr int kSmem = kGroups * kSmemGroup;
  static constexpr int kPerSm = 2;  // resident CTAs per SM
};

template <int kMA, int kNB, bool kDiag, int kG>
__global__ void __launch_bounds__(NtkShape<kMA, kNB, kDiag, kG>::kThr, NtkShape<kMA, kNB, kDiag, kG>::kPerSm)
k_f32_ntk(const float* __restrict__ G, int64_t gstride, int B, const __grid_constant__ NtkParts parts, double* part, uint32_t* done,
          float* __restrict__ K) {
  pdl_wait();
  typedef NtkShape<kMA, kNB, kDiag, kG> S;
  extern __shared__ __align__(16) float smem_cta[];
  const int group = threadIdx.x / kNtkThreads, tid = threadIdx.x % kNtkThreads, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  float* smem = smem_cta + group * (S::kSmemGroup / 4);
  auto sync_group = [&]() {
    if (S::kGroups == 1) __syncthreads();
    else asm volatile("bar.sync %0, %1;" ::"r"(group + 1), "n"(kNtkThreads) : "memory");
  };
  const int64_t first_chunk = (int64_t)blockIdx.y * S::kGroups + group, chunk_step = (int64_t)gridDim.y * S::kGroups;
  int i0, j0;
  ntk_pair_rows(kDiag, blockIdx.x, i0, j0);
  const int64_t nchunks = (gstride + kNtkKC - 1) / kNtkKC;
  auto fetch = [&](int64_t ch, int stage) {
    if (ch < nchunks) {
      float* s = smem + stage * S::kStageFloats;
      for (int e = tid; e < S::kRowsStaged * (kNtkKC / 4); e += kNtkThreads) {
        const int r = e / (kNtkKC / 4), c = e % (kNtkKC / 4) * 4;
        const int seq = kDiag || r < 16 * kMA ? i0 + r : j0 + r - 16 * kMA;
        const int64_t x = ch * kNtkKC + c;
        const bool live = seq < B && x < gstride;
        cp_async16(s + r * kNtkPitch + c, live ? G + (size_t)seq * gstride + x : G, live);
      }
    }
    cp_async_commit();
  };
  double acc[kMA][kNB][4];
#pragma unroll
  for (int p = 0; p < kMA; ++p)
#pragma unroll
    for (int n = 0; n < kNB; ++n)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[p][n][q] = 0.0;
#pragma unroll
  for (int k = 0; k < kNtkStages - 1; ++k) fetch(first_chunk + k * chunk_step, k);
  int stage = 0;
  for (int64_t ch = first_chunk; ch < nchunks; ch += chunk_step) {
    cp_async_wait<kNtkStages - 2>();
    sync_group();
    fetch(ch + (kNtkStages - 1) * chunk_step, (stage + kNtkStages - 1) % kNtkStages);
    const float* s = smem + stage * S::kStageFloats;
    if (++stage == kNtkStages) stage = 0;
#pragma unroll
    for (int h = 0; h < kNtkKC / 32; ++h) {
      const int k0 = (warp + 4 * h) * 8 + t;
      double b[kNB][2];
      const float* sb = s + (kDiag ? 0 : 16 * kMA) * kNtkPitch;
#pragma unroll
      for (int n = 0; n < kNB; ++n) {
        b[n][0] = (double)sb[(n * 8 + g) * kNtkPitch + k0];
        b[n][1] = (double)sb[(n * 8 + g) * kNtkPitch + k0 + 4];
      }
#pragma unroll
      for (int p = 0; p < kMA; ++p) {
        double a0, a1, a2, a3;
        if (kDiag) {  // rows and columns are the same sequences, and a fragment of either holds the same elements
          a0 = b[2 * p][0]; a1 = b[2 * p + 1][0]; a2 = b[2 * p][1]; a3 = b[2 * p + 1][1];
        } else {
          a0 = (double)s[(p * 16 + g) * kNtkPitch + k0];
          a1 = (double)s[(p * 16 + 8 + g) * kNtkPitch + k0];
          a2 = (double)s[(p * 16 + g) * kNtkPitch + k0 + 4];
          a3 = (double)s[(p * 16 + 8 + g) * kNtkPitch + k0 + 4];
        }
#pragma unroll
        for (int n = kDiag ? 2 * p : 0; n < kNB; ++n) dmma16x8x8(acc[p][n], a0, a1, a2, a3, b[n][0], b[n][1]);
      }
    }
  }
  cp_async_wait<0>();
  // the warps' shares meet in shared memory (4 -> 2 -> 1)
  double2* red = reinterpret_cast<double2*>(smem);
  for (int half = 2; half >= 1; half >>= 1) {
    sync_group();
    if (warp >= half && warp < 2 * half) {
      int blk = (warp - half) * S::kBlocks;
#pragma unroll
      for (int p = 0; p < kMA; ++p)
#pragma unroll
        for (int n = kDiag ? 2 * p : 0; n < kNB; ++n, ++blk) {
          red[blk * 64 + lane] = make_double2(acc[p][n][0], acc[p][n][1]);
          red[blk * 64 + 32 + lane] = make_double2(acc[p][n][2], acc[p][n][3]);
        }
    }
    sync_group();
    if (warp < half) {
      int blk = warp * S::kBlocks;
#pragma unroll
      for (int p = 0; p < kMA; ++p)
#pragma unroll
        for (int n = kDiag ? 2 * p : 0; n < kNB; ++n, ++blk) {
          const double2 lo = red[blk * 64 + lane], hi = red[blk * 64 + 32 + lane];
          acc[p][n][0] += lo.x; acc[p][n][1] += lo.y; acc[p][n][2] += hi.x; acc[p][n][3] += hi.y;
        }
    }
  }
  if (S::kGroups > 1) {  // the groups' shares, in order
    __syncthreads();
    double* meet = reinterpret_cast<double*>(smem_cta) + lane;  // [group - 1][kBlocks][4][32]
    if (group > 0 && warp == 0) {
      double* to = meet + (group - 1) * S::kBlocks * 128;
#pragma unroll
      for (int p = 0; p < kMA; ++p)
#pragma unroll
        for (int n = kDiag ? 2 * p : 0; n < kNB; ++n)
#pragma unroll
          for (int q = 0; q < 4; ++q, to += 32) *to = acc[p][n][q];
    }
    __syncthreads();
    if (group == 0 && warp == 0) {
      for (int k = 0; k < S::kGroups - 1; ++k) {
        const double* from = meet + k * S::kBlocks * 128;
#pragma unroll
        for (int p = 0; p < kMA; ++p)
#pragma unroll
          for (int n = kDiag ? 2 * p : 0; n < kNB; ++n)
#pragma unroll
            for (int q = 0; q < 4; ++q, from += 32) acc[p][n][q] += *from;
      }
    }
  }
  static_assert((S::kGroups - 1) * S::kBlocks * 128 * 8 <= S::kSmem, "the groups' shares");
  // k_f32_ntk_finish is set up while the shares of a single pair are stored (of several pairs it is larger, and slower so)
  if (kDiag && gridDim.x == 1 && !done) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (group == 0 && warp == 0) {
    double* mine = part + ((int64_t)blockIdx.x * gridDim.y + blockIdx.y) * parts.doubles + lane;
#pragma unroll
    for (int p = 0; p < kMA; ++p)
#pragma unroll
      for (int n = kDiag ? 2 * p : 0; n < kNB; ++n)
#pragma unroll
        for (int q = 0; q < 4; ++q, mine += 32)
          if (i0 + p * 16 + (q >> 1) * 8 < B && j0 + n * 8 < B) *mine = acc[p][n][q];  // others stand for no sequences: never read
  }
  if (done) {  // one pair, few shares
    // an entry of K to a thread, or, of many shares, to as many threads as there are for each, which meet in shared memory
    const int entries = B * (B + 1) / 2, shares = (int)gridDim.y, runs = shares <= 16 ? 1 : S::kThr / entries;
    const int mine = runs > 1 ? threadIdx.x / runs : threadIdx.x;
    int i, j;
    int x = ntk_triangle(parts, B, min(mine, entries - 1), i, j);
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(done, 1u) == gridDim.y - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    if (runs <= 1) {
      for (int e = mine; e < entries; e += 2 * S::kThr) {  // two at a time
        int i1, j1;
        const int e1 = e + S::kThr, x1 = e1 < entries ? ntk_triangle(parts, B, e1, i1, j1) : 0;
        if (e != mine) x = ntk_triangle(parts, B, e, i, j);
        double v[8], v1[8], t0 = 0.0, t1 = 0.0;
        for (int k = 0; k < shares; k += 8) {
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            v[u] = k + u < shares ? __ldcg(part + (int64_t)(k + u) * parts.doubles + x) : 0.0;
            v1[u] = k + u < shares && e1 < entries ? __ldcg(part + (int64_t)(k + u) * parts.doubles + x1) : 0.0;
          }
          t0 += ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
          t1 += ((v1[0] + v1[1]) + (v1[2] + v1[3])) + ((v1[4] + v1[5]) + (v1[6] + v1[7]));
        }
        ntk_write(K, B, i, j, t0);
        if (e1 < entries) ntk_write(K, B, i1, j1, t1);
      }
      return;
    }
    const int run = threadIdx.x % runs, per = (shares + runs - 1) / runs, first = min(shares, run * per);
    double* sums = reinterpret_cast<double*>(smem_cta);
    sums[threadIdx.x] = ntk_sum<16>(part + x, parts.doubles, first, min(shares, first + per));
    __syncthreads();
    if (mine >= entries || run != 0) return;
    double v = 0.0;
    for (int k = 0; k < runs; ++k) v += sums[threadIdx.x + k];
    ntk_write(K, B, i, j, v);
  }
}

// K from the shares of a launch on the diagonal blocks and, with more than one of them, of one on the others.  The shares of an
// element are added in kRuns runs, a thread each, so that a thread's loads are no long chain: one run where shares are few (up to
// 16), 8 or, above 128 shares (there are 296 at most), 32: a thread's loads are all in flight at once.
template <int kRuns>
__global__ void __launch_bounds__(256) k_f32_ntk_finish(const __grid_constant__ NtkParts diag, const __grid_constant__ NtkParts rest,
                                                        const double* __restrict__ part, int B, float* __restrict__ K) {
  pdl_wait();
  constexpr int kElems = 256 / kRuns;  // of a block
  __shared__ double sums[kRuns][kElems];
  const int t = threadIdx.x % kElems, run = threadIdx.x / kElems;
  const int64_t diag_blocks = diag.pairs * diag.doubles / kElems;
  const bool on_diag = blockIdx.x < diag_blocks;
  const NtkParts& P = on_diag ? diag : rest;
  const int64_t x = (on_diag ? blockIdx.x : blockIdx.x - diag_blocks) * kElems;
  const int64_t pair = x / P.doubles;
  const int e = (int)(x - pair * P.doubles) + t;
  int i0, j0, i, j;
  ntk_pair_rows(P.diag, pair, i0, j0);
  const bool used = ntk_entry(P, i0, j0, e, B, i, j);
  const double* src = part + (on_diag ? 0 : diag.total()) + pair * P.slabs * P.doubles + e;
  const int per = (int)((P.slabs + kRuns - 1) / kRuns), first = min((int)P.slabs, run * per);
  double s = used ? ntk_sum<16>(src, P.doubles, first, min((int)P.slabs, first + per)) : 0.0;
  if (kRuns > 1) {
    sums[run][t] = s;
    __syncthreads();
    if (run != 0) return;
    s = 0.0;
#pragma unroll
    for (int w = 0; w < kRuns; ++w) s += sums[w][t];
  }
  if (used) ntk_write(K, B, i, j, s);
}

// ---------------------------------------------------------------------------------------------
// Products over token pairs: for a kGT x kGT tile (row tokens x column tokens) P = RX X^T and Q = RY dY^T, multiplied
// elementwise and summed per (row segment, column sequence) in float64.  Operand rows are staged 16 features at a time
// by cp.async and read four features at once (16-byte shared loads, rows 20 floats apart: no bank conflicts); an element
// is a sum over the even and one over the odd features, the two halves of a packed fma.
//   Gram (kSampled = false): rows and columns are both tokens, tile pairs I <= J.  Only token pairs t <= s are used; a
//     pair inside one sequence with t < s stands for (t,s) and (s,t) and counts twice.
//   Sampled estimator (kSampled = true): the rows are the gathered sample rows, out = M^T[sample, sequence], no weights.
// The tile's products go through shared memory; a warp owns 32 rows of some columns of them, walks the columns (sequence
// boundaries are the same for all its lanes), and adds the lanes of one row sequence together before it issues one
// float64 atomic.  Bound by the float32 pipe and, with few CTAs on an SM, by the latency of a stage.  Tiles of 64 have 8 x 4 elements a
// thread, two thirds of the shared-memory reads of 4 x 4, and 128 threads whose registers and memory let three CTAs share an SM (two of
// 256 threads before): 896 -> 896, 4608 tokens 1140 -> 1000 us; 128 samples of 20000 332 -> 291, 7032 tokens 1481 x 1513 236 -> 196.
// Too few tiles of 64 to fill the machine leave the kernel to the latency of one CTA's walk over the features: tiles of 32 then, and
// clusters of kC CTAs that take a share of the features each and add up their sums through distributed shared memory before P and Q
// are multiplied (f32_gram_shape); those have the registers to load ahead (72 a thread -> 132: 450 tokens, 1536 x 1536 60 -> 53 us).
// The pairs I <= J are numbered in one row: of a square grid of which half returns at once some SMs got three times the work of
// others (789 tokens, 251 x 1121 97 -> 74 us).
// ---------------------------------------------------------------------------------------------
constexpr int kGK = 16;   // features per stage
constexpr int kGPitch = kGK + 4;

template <int kGT>
struct GramTile {
  static constexpr int kRows = kGT == 64 ? 8 : 2, kCols = 4;        // elements of a thread
  static constexpr int kTx = kGT / kCols, kTy = kGT / kRows;        // 64: 8 x 16 threads; 32: 16 x 8
  static constexpr int kStages = kGT == 64 ? 3 : 6;                 // 30 KB either way
};
__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ float ld_cluster(const float* mine, unsigned rank) {  // what CTA `rank` has where this one has *mine
  uint32_t at;
  float v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"((uint32_t)__cvta_generic_to_shared(mine)), "r"(rank));
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(at) : "memory");
  return v;
}
template <bool kSampled, int kGT, int kC>
__global__ void __launch_bounds__(128, kGT == 64 ? 3 : kC == 1 ? 7 : 2) k_f32_gram(const float* __restrict__ RX, const float* __restrict__ RY, int64_t n_rows,
                                                  const float* __restrict__ X, const float* __restrict__ dY, int64_t T,
                                                  int d_in, int d_out, const int32_t* __restrict__ tokseq, int B,
                                                  double* __restrict__ out) {
  pdl_wait();
  constexpr int kRows = GramTile<kGT>::kRows, kTx = GramTile<kGT>::kTx, kTy = GramTile<kGT>::kTy, kThr = kTx * kTy;
  static_assert(kThr == 128, "threads");
  constexpr int kGramStages = GramTile<kGT>::kStages;
  const unsigned rank = kC > 1 ? cluster_rank() : 0, unit = blockIdx.x / kC;
  int I, J;
  if (kSampled) {
    const unsigned ns = (unsigned)((n_rows + kGT - 1) / kGT);
    J = (int)(unit / ns);
    I = (int)(unit - (unsigned)J * ns);
  } else {  // tile column J has tiles 0 .. J
    J = (int)((sqrt(8.0 * unit + 1.0) - 1.0) * 0.5);
    while ((int64_t)J * (J + 1) / 2 > unit) --J;
    while ((int64_t)(J + 1) * (J + 2) / 2 <= unit) ++J;
    I = (int)(unit - (int64_t)J * (J + 1) / 2);
  }
  constexpr int kStageFloats = kGramStages * 2 * kGT * kGPitch, kTile = kGT * (kGT + 1);
  // The sums of Q go where the stages were, [row][kGT + 1]; those of P behind them, from tiles of 64 as soon as P's features are
  // done (they would take 32 registers).
  constexpr bool kParkP = kGT == 64;
  static_assert(kParkP ? kTile <= kStageFloats : 2 * kTile <= kStageFloats, "shared memory");
  __shared__ __align__(16) float smem[kStageFloats + (kParkP ? kTile : 0)];
  float* const tile_q = smem;
  float* const tile_p = smem + (kParkP ? kStageFloats : kTile);
  auto stage_mem = [&](int k, int side) { return smem + (k % kGramStages * 2 + side) * (kGT * kGPitch); };
  __shared__ int s_col[kGT];
  const int tid = threadIdx.x, tx = tid % kTx, ty = tid / kTx;
  const int64_t r0 = (int64_t)I * kGT, c0 = (int64_t)J * kGT;
  if (tid < kGT) s_col[tid] = c0 + tid < T ? tokseq[c0 + tid] : -1;
  const int nkx = (d_in + kGK - 1) / kGK, total_k = nkx + (d_out + kGK - 1) / kGK;
  const int k0 = (int)((int64_t)total_k * rank / kC), k1 = (int)((int64_t)total_k * (rank + 1) / kC);  // this CTA's stages
  // a thread copies one column (group) of a stage, every kThr / kGK-th (4-byte copies) or 4 kThr / kGK-th row
  const int c1 = tid % kGK, r1 = tid / kGK, c4 = tid % (kGK / 4) * 4, r4 = tid / (kGK / 4);
  auto fetch = [&](int k) {
    if (k < k1) {
      const bool second = k >= nkx;
      const int d = second ? d_out : d_in, f0 = (second ? k - nkx : k) * kGK;
#pragma unroll
      for (int side = 0; side < 2; ++side) {
        const float* M = side == 0 ? (second ? RY : RX) : (second ? dY : X);
        const int64_t first = side == 0 ? r0 : c0;
        const int rows = (int)min((int64_t)kGT, (side == 0 ? n_rows : T) - first);  // rows of the tile that exist
        float* dst = stage_mem(k - k0, side);
        if ((d & 3) == 0) {
          const float* src = M + (first + r4) * d + f0 + c4;
#pragma unroll
          for (int i = 0; i < kGT; i += 4 * kThr / kGK, src += (int64_t)(4 * kThr / kGK) * d) {
            const bool live = r4 + i < rows && f0 + c4 < d;
            cp_async16(dst + (r4 + i) * kGPitch + c4, live ? src : M, live);
          }
        } else {
          const float* src = M + (first + r1) * d + f0 + c1;
#pragma unroll
          for (int i = 0; i < kGT; i += kThr / kGK, src += (int64_t)(kThr / kGK) * d) {
            const bool live = r1 + i < rows && f0 + c1 < d;
            cp_async4(dst + (r1 + i) * kGPitch + c1, live ? src : M, live);
          }
        }
      }
    }
    cp_async_commit();
  };
  float h[kParkP ? 1 : kRows][4] = {};
  f32x2 acc[kRows][4] = {};
  auto place = [&](int p, int q) { return (ty + kTy * p) * (kGT + 1) + tx + kTx * q; };
  auto total = [](f32x2 v) { float lo, hi; unpack2(v, lo, hi); return lo + hi; };
  auto keep_p = [&]() {  // the sums so far are of P
#pragma unroll
    for (int p = 0; p < kRows; ++p)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float v = total(acc[p][q]);
        if (kParkP) tile_p[place(p, q)] = v;
        else h[kParkP ? 0 : p][q] = v;
        acc[p][q] = 0ull;
      }
  };
  for (int k = k0; k < k0 + kGramStages - 1; ++k) fetch(k);
  if (kC > 1 && kParkP && k0 > nkx) keep_p();  // no features of P here: zeros
  for (int k = k0; k < k1; ++k) {
    cp_async_wait<kGramStages - 2>();
    __syncthreads();
    fetch(k + kGramStages - 1);
    if (k == nkx) keep_p();
    const float* sA = stage_mem(k - k0, 0);
    const float* sB = stage_mem(k - k0, 1);
#pragma unroll
    for (int c = 0; c < kGK; c += 4) {
      ulonglong2 a[kRows], b[4];
#pragma unroll
      for (int p = 0; p < kRows; ++p) a[p] = *reinterpret_cast<const ulonglong2*>(sA + (ty + kTy * p) * kGPitch + c);
#pragma unroll
      for (int q = 0; q < 4; ++q) b[q] = *reinterpret_cast<const ulonglong2*>(sB + (tx + kTx * q) * kGPitch + c);
#pragma unroll
      for (int p = 0; p < kRows; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[p][q] = fma2(a[p].y, b[q].y, fma2(a[p].x, b[q].x, acc[p][q]));
    }
  }
  cp_async_wait<0>();
  __syncthreads();
  if (k1 <= nkx) keep_p();
  // One CTA: the products.  Several: the sums of P and behind them those of Q, which every CTA of the cluster reads for its share
  // of the columns and adds up in rank order.
#pragma unroll
  for (int p = 0; p < kRows; ++p)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int e = place(p, q);
      const float y = total(acc[p][q]), x = kParkP ? (kC == 1 ? tile_p[e] : 0.0f) : h[kParkP ? 0 : p][q];
      tile_q[e] = kC == 1 ? x * y : y;
      if (kC > 1 && !kParkP) tile_p[e] = x;
    }
  if (kC == 1) __syncthreads();
  else cluster_sync();
  // a warp takes 32 rows and kWidth columns
  constexpr int kWarpCols = 4 / (kGT / 32), kWidth = kGT / kWarpCols / kC;  // warps side by side
  const int warp = tid >> 5, lane = tid & 31, row = (warp % (kGT / 32)) * 32 + lane, cb = (int)(rank * kWarpCols + warp / (kGT / 32)) * kWidth;
  const int mine = row * (kGT + 1) + cb;
  float prod[kWidth];
  if (kC > 1) {  // all of the loads in flight together
    float x[kC][kWidth], y[kC][kWidth];
#pragma unroll
    for (int r = 0; r < kC; ++r)
#pragma unroll
      for (int c = 0; c < kWidth; ++c) { x[r][c] = ld_cluster(tile_p + mine + c, r); y[r][c] = ld_cluster(tile_q + mine + c, r); }
#pragma unroll
    for (int c = 0; c < kWidth; ++c) {
      float sx = x[0][c], sy = y[0][c];
#pragma unroll
      for (int r = 1; r < kC; ++r) { sx += x[r][c]; sy += y[r][c]; }
      prod[c] = sx * sy;
    }
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");  // this CTA has read the others' sums
  } else {
#pragma unroll
    for (int c = 0; c < kWidth; ++c) prod[c] = tile_q[mine + c];
  }
  const int64_t t = r0 + row;
  const int rseq = t < n_rows ? (kSampled ? (int)t : tokseq[t]) : -1;  // rows past the end form a run of their own, unused
  int same = 0;
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    const int other = __shfl_down_sync(0xffffffffu, rseq, 1 << k);
    if (lane + (1 << k) < 32 && other == rseq) same |= 1 << k;
  }
  const int up = __shfl_up_sync(0xffffffffu, rseq, 1);
  const bool head = (lane == 0 || up != rseq) && rseq >= 0;
  double run = 0.0;
#pragma unroll
  for (int c = 0; c < kWidth; ++c) {
    const int cs = s_col[cb + c];
    if (cs < 0) break;
    const int64_t s = c0 + cb + c;
    const double v = (double)prod[c];
    if (kSampled) run += v;
    else if (t <= s) run += rseq == cs && t < s ? 2.0 * v : v;
    if (c == kWidth - 1 || s_col[cb + c + 1] != cs) {
#pragma unroll
      for (int k = 0; k < 5; ++k) {
        const double o = __shfl_down_sync(0xffffffffu, run, 1 << k);
        if ((same >> k) & 1) run += o;
      }
      if (head && run != 0.0) atomicAdd(&out[(size_t)rseq * B + cs], run);
      run = 0.0;
    }
  }
  if (kC > 1) {
    __syncwarp();  // the barrier wants the warp together
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");  // nobody leaves while its sums may still be read
  }
}

__global__ void k_f32_gram_finish(const double* __restrict__ kacc, int B, float* __restrict__ K) {
  pdl_wait();
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= (int64_t)B * B) return;
  const int i = (int)(e / B), j = (int)(e % B);
  K[e] = (float)(i <= j ? kacc[(size_t)i * B + j] : kacc[(size_t)j * B + i]);
}

// dW = beta dW + sum_i c_i G_i, four elements per lane, eight 16-byte loads in flight, float64 sums.  HBM stream: 205 MB in
// 29 us against 60 us with one 4-byte load per thread and sequence.  As in the bf16 combine a small layer splits the
// sequences over the warps of a block (kSlices of them) and adds the shares in shared memory: 300 x 500 at 256 sequences
// 28 us split, 120 us whole.
template <int kSlices>
__global__ void __launch_bounds__(256) k_f32_combine(const float* __restrict__ G, int64_t N, int64_t gstride, int B,
                                                     const float* __restrict__ coeffs, float* __restrict__ dW, float beta,
                                                     const WsTag* __restrict__ tag_dev, WsTag tag,
                                                     int32_t* __restrict__ info) {
  pdl_wait();
  if (!ws_tag_matches(tag_dev, tag, info)) return;
  constexpr int kLanes = 256 / kSlices;
  __shared__ double4 part[kSlices > 1 ? 256 : 1];
  const int x = threadIdx.x % kLanes, slice = threadIdx.x / kLanes;
  const int per = (B + kSlices - 1) / kSlices, i1 = min(B, (slice + 1) * per);
  for (int64_t e0 = 4 * (int64_t)blockIdx.x * kLanes; e0 < N; e0 += 4 * (int64_t)gridDim.x * kLanes) {
    const int64_t e = e0 + 4 * x;
    double4 s = make_double4(0.0, 0.0, 0.0, 0.0);
    auto add = [&](const float4& v, float c) {
      s.x += (double)c * (double)v.x; s.y += (double)c * (double)v.y;
      s.z += (double)c * (double)v.z; s.w += (double)c * (double)v.w;
    };
    const float* src = G + e;
    int i = e < N ? slice * per : i1;
    for (; i + 8 <= i1; i += 8) {
      float4 v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = __ldcs(reinterpret_cast<const float4*>(src + (size_t)(i + u) * gstride));
#pragma unroll
      for (int u = 0; u < 8; ++u) add(v[u], __ldg(coeffs + i + u));
    }
    for (; i < i1; ++i) add(__ldcs(reinterpret_cast<const float4*>(src + (size_t)i * gstride)), __ldg(coeffs + i));
    if (kSlices > 1) {
      part[threadIdx.x] = s;
      __syncthreads();
      if (slice == 0)
#pragma unroll
        for (int k = 1; k < kSlices; ++k) {
          const double4 o = part[k * kLanes + x];
          s.x += o.x; s.y += o.y; s.z += o.z; s.w += o.w;
        }
      __syncthreads();
      if (slice != 0) continue;
    }
    const double v[4] = {s.x, s.y, s.z, s.w};
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (e + k < N) dW[e + k] = (float)(beta != 0.f ? (double)dW[e + k] + v[k] : v[k]);
  }
}

}  // namespace

template <int kOut>
static isopo_status prep(const int64_t* off_host, int B, int64_t T, int64_t* off_dev, const float* coeffs, void* out,
                         const Clear& clear, cudaStream_t st) {
  const int64_t work = std::max<int64_t>(kOut == kOffsetsOnly ? 1 : T, (clear.n[0] + clear.n[1] + clear.n[2]) / 4);
  const int grid = (int)std::min<int64_t>((work + 255) / 256, 1184);
  LaunchScope scope(kIdPrep, st);
  if (B + 1 <= kArgChunk) {
    OffsetArgs<kArgChunk> a;
    fill_offsets(&a, off_host, B + 1);
    launch(k_prep<kOut, kArgChunk>, grid, 256, 0, st, a, B, T, off_dev, coeffs, out, clear);
  } else if (B + 1 <= kArgLarge) {
    OffsetArgs<kArgLarge> a;
    fill_offsets(&a, off_host, B + 1);
    launch(k_prep<kOut, kArgLarge>, grid, 256, 0, st, a, B, T, off_dev, coeffs, out, clear);
  } else {
    for (int64_t base = 0; base <= B; base += kArgLarge) {
      OffsetArgs<kArgLarge> a;
      const int m = (int)std::min<int64_t>(kArgLarge, B + 1 - base);
      fill_offsets(&a, off_host + base, m);
      launch(k_store_offsets<kArgLarge>, 1, 256, 0, st, a, base, m, off_dev);
    }
    ISOPO_CUDA_TRY(cudaGetLastError());
    if (kOut != kOffsetsOnly || clear.n[0] + clear.n[1] + clear.n[2] > 0)
      launch(k_prep_many<kOut>, grid, 256, 0, st, off_dev, B, T, coeffs, out, clear);
  }
  ISOPO_CUDA_TRY(cudaGetLastError());
  return ISOPO_OK;
}

isopo_status launch_prep(const int64_t* off_host, int B, int64_t T, int64_t* off_dev, int32_t* tokseq, const Clear& clear,
                         cudaStream_t st) {
  return prep<kTokSeq>(off_host, B, T, off_dev, nullptr, tokseq, clear, st);
}

isopo_status launch_prep_repitch(const int64_t* off_host, int B, int64_t T, int64_t* off_dev, int32_t* tokseq, const Clear& clear,
                                 const Repitch& repitch, cudaStream_t st) {
  const int64_t work = std::max<int64_t>(32 * T, (clear.n[0] + clear.n[1] + clear.n[2]) / 4);
  const int grid = (int)std::min<int64_t>((work + 255) / 256, 1184);
  LaunchScope scope(kIdPrep, st);
  auto with_args = [&](auto kernel, auto* a) {
    fill_offsets(a, off_host, B + 1);
    launch(kernel, grid, 256, 0, st, *a, B, T, off_dev, tokseq, clear, repitch);
  };
  if (B + 1 <= kArgChunk) {
    OffsetArgs<kArgChunk> a;
    with_args(k_prep_repitch<kArgChunk>, &a);
  } else {
    OffsetArgs<kArgLarge> a;
    with_args(k_prep_repitch<kArgLarge>, &a);
  }
  ISOPO_CUDA_TRY(cudaGetLastError());
  return ISOPO_OK;
}
isopo_status launch_tokscale(const int64_t* off_host, int B, int64_t T, int64_t* off_dev, const float* coeffs,
                             float* tokscale, const Clear& clear, cudaStream_t st) {
  return prep<kTokScale>(off_host, B, T, off_dev, coeffs, tokscale, clear, st);
}

isopo_status launch_offsets(const int64_t* off_host, int B, int64_t* off_dev, const Clear& clear, cudaStream_t st) {
  return prep<kOffsetsOnly>(off_host, B, 0, off_dev, nullptr, nullptr, clear, st);
}

void make_stored_intake(StoredIntake* a, const int64_t* off_host, int B, int n_proj, const WsTag* tag, WsHead* const* head,
                        float* const* acc, int n_acc) {
  for (int i = 0; i <= B; ++i) a->off[i] = (int32_t)off_host[i];
  a->n_proj = n_proj;
  a->n_acc = n_acc;
  for (int h = 0; h < 3; ++h) {
    const int hh = h < n_proj ? h : 0;
    a->tag[h] = tag[hh]; a->head[h] = head[hh]; a->acc[h] = acc[hh];
  }
  // longest first; equal lengths keep their order: sort (complement of the length, index)
  uint64_t key[256];
  for (int i = 0; i < B; ++i) key[i] = ((uint64_t)(~(uint32_t)(a->off[i + 1] - a->off[i])) << 32) | (uint32_t)i;
  std::sort(key, key + B);
  for (int i = 0; i < B; ++i) a->order[i] = (uint8_t)key[i];
}

template <int kTile, int kT, bool kArgOff>
static isopo_status launch_f32_seq_grad(const F32StoredArgs& a, const OffsetParam<kArgOff>& o, cudaStream_t st) {
  typedef SeqGemm<kTile, kT> Gemm;
  const dim3 grid((a.d_in + kTile - 1) / kTile, (a.d_out + kTile - 1) / kTile, a.B);
  if (grid.y > 65535 || grid.z > 65535) return ISOPO_ERR_UNSUPPORTED;
  ISOPO_CUDA_TRY(cudaFuncSetAttribute(k_f32_seq_grad<kTile, kT, kArgOff>, cudaFuncAttributeMaxDynamicSharedMemorySize, Gemm::kSmem));
  {
    LaunchScope scope(kIdF32SeqGrad, st);
    launch(k_f32_seq_grad<kTile, kT, kArgOff>, grid, Gemm::kThr, Gemm::kSmem, st, a, o);
  }
  ISOPO_CUDA_TRY(cudaGetLastError());
  return ISOPO_OK;
}

// 128 x 128 tiles (8 x 8 per thread) where they fill the machine twice and pad little, else 64 x 64 (4 x 4).
static bool f32_wide_tiles(int d_in, int d_out, int64_t copies) {
  const int64_t gx = (d_in + 127) / 128, gy = (d_out + 127) / 128, hx = (d_in + 63) / 64, hy = (d_out + 63) / 64;
  return gx * gy * copies >= 2 * kSms && gx * gy * 4 * 4 <= hx * hy * 5;
}

isopo_status f32_seq_grad(const float* X, const float* dY, int d_in, int d_out, const int64_t* off_host, int64_t* off_dev,
                          int B, float* G, int64_t gstride, uint32_t* done, const WsTag& tag, WsTag* tag_dev, cudaStream_t st) {
  F32StoredArgs a{X, dY, d_in, d_out, B, gstride, off_dev, G, done, tag, tag_dev};
  const bool wide = f32_wide_tiles(d_in, d_out, B);
  if (B + 1 <= kArgChunk) {
    OffsetParam<true> o;
    for (int i = 0; i <= B; ++i) o.v[i] = (int32_t)off_host[i];
    return wide ? launch_f32_seq_grad<128, 8, true>(a, o, st) : launch_f32_seq_grad<64, 4, true>(a, o, st);
  }
  isopo_status s = launch_offsets(off_host, B, off_dev, Clear{}, st);
  if (s != ISOPO_OK) return s;
  const OffsetParam<false> o{};
  return wide ? launch_f32_seq_grad<128, 8, false>(a, o, st) : launch_f32_seq_grad<64, 4, false>(a, o, st);
}

// groups: of four warps in a CTA; at least eight chunks to a CTA of one group, or the reduction outweighs the stream
static NtkParts ntk_parts(int ma, int nb, bool diag, int groups, int64_t chunks, int64_t pairs) {
  const int64_t ctas = 2 * kSms, least = groups == 1 ? 8 : 4 * groups;  // every SM full over all pairs
  const int64_t slabs = std::max<int64_t>(1, std::min<int64_t>((ctas + pairs - 1) / pairs, (chunks + least - 1) / least));
  return NtkParts{pairs, slabs, ma, nb, ntk_blocks(ma, nb, diag) * 128, groups, diag};
}
// The launches of the K pass of B gradients: diagonal blocks, the others (no pairs: none).  Up to 32 sequences two CTAs of one
// group on every SM where that gives a group sixteen chunks or fewer, else two of several.
static void ntk_plan(int64_t gstride, int B, NtkParts* diag, NtkParts* rest) {
  const int64_t blocks = (B + kNtkRows - 1) / kNtkRows, chunks = (gstride + kNtkKC - 1) / kNtkKC;
  const bool few_chunks = chunks <= 16 * 2 * kSms;
  *diag = B <= 16   ? ntk_parts(1, 2, true, few_chunks ? 1 : 4, chunks, 1)
          : B <= 32 ? ntk_parts(2, 4, true, few_chunks ? 1 : 2, chunks, 1)
                    : ntk_parts(4, 8, true, 1, chunks, blocks);
  *rest = blocks == 1 ? NtkParts{} : ntk_parts(2, 8, false, 1, chunks, blocks * (blocks - 1));  // two halves of that many / 2 pairs
}
size_t f32_ntk_part_bytes(int64_t gstride, int B) {
  NtkParts diag, rest;
  ntk_plan(gstride, B, &diag, &rest);
  return sizeof(double) * (size_t)(diag.total() + rest.total());
}

template <int kMA, int kNB, bool kDiag, int kG>
static isopo_status launch_f32_ntk(const float* G, int64_t gstride, int B, const NtkParts& parts, double* part, uint32_t* done,
                                   float* K, cudaStream_t st) {
  typedef NtkShape<kMA, kNB, kDiag, kG> S;
  const auto kernel = k_f32_ntk<kMA, kNB, kDiag, kG>;
  ISOPO_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, S::kSmem));
  {
    LaunchScope scope(kIdF32Ntk, st);
    launch(kernel, dim3((unsigned)parts.pairs, (unsigned)parts.slabs), S::kThr, S::kSmem, st, G, gstride, B, parts, part, done, K);
  }
  ISOPO_CUDA_TRY(cudaGetLastError());
  return ISOPO_OK;
}

static isopo_status launch_f32_finish(const double* kacc, int B, float* K, cudaStream_t st) {
  {
    LaunchScope scope(kIdMirror, st);
    launch(k_f32_gram_finish, (unsigned)(((int64_t)B * B + 255) / 256), 256, 0, st, kacc, B, K);
  }
  ISOPO_CUDA_TRY(cudaGetLastError());
  return ISOPO_OK;
}

isopo_status f32_ntk(const float* G, int64_t gstride, int B, double* part, uint32_t* done, float* K, cudaStream_t st) {
  NtkParts diag, rest;
  ntk_plan(gstride, B, &diag, &rest);
  // The last CTA adds the shares up itself, a launch less, where that takes it about as long as one round of loads: its threads
  // are several to an entry of K, or have no more than two rounds of two entries.
  const int threads = kNtkThreads * diag.groups, entries = B <= kNtkRows ? B * (B + 1) / 2 : INT32_MAX;
  const bool by_last = diag.pairs == 1 && (threads >= 2 * entries ? diag.slabs <= 48 * (threads / entries)
                                                                  : (entries + 2 * threads - 1) / (2 * threads) * ((diag.slabs + 7) / 8) <= 2);
  if (!by_last) done = nullptr;
  const auto launch_diag = B <= 16   ? (diag.groups == 1 ? launch_f32_ntk<1, 2, true, 1> : launch_f32_ntk<1, 2, true, 4>)
                           : B <= 32 ? (diag.groups == 1 ? launch_f32_ntk<2, 4, true, 1> : launch_f32_ntk<2, 4, true, 2>)
                                     : launch_f32_ntk<4, 8, true, 1>;
  const isopo_status s = launch_diag(G, gstride, B, diag, part, done, K, st);
  if (s != ISOPO_OK || by_last) return s;
  if (rest.pairs > 0) {
    const isopo_status r = launch_f32_ntk<2, 8, false, 1>(G, gstride, B, rest, part + diag.total(), nullptr, K, st);
    if (r != ISOPO_OK) return r;
  }
  {
    LaunchScope scope(kIdMirror, st);
    const int64_t shares = std::max(diag.slabs, rest.slabs), elems = diag.pairs * diag.doubles + rest.pairs * rest.doubles;
    const int runs = shares > 128 ? 32 : shares > 16 ? 8 : 1;
    launch(runs == 32 ? k_f32_ntk_finish<32> : runs == 8 ? k_f32_ntk_finish<8> : k_f32_ntk_finish<1>,
           (unsigned)(elems * runs / 256), 256, 0, st, diag, rest, part, B, K);  // elems: a multiple of 256
  }
  ISOPO_CUDA_TRY(cudaGetLastError());
  return ISOPO_OK;
}

// Tokens per tile and CTAs that share a tile's features.  Few tiles of 32: as many CTAs to each as make up to 240 of them, as one alone
// is a chain of (d_in + d_out) / 16 stages.  Else tiles of 32, of 64, or of 64 by two CTAs, whichever costs least: us per stage with k
// CTAs on an SM, a constant, and for two CTAs the exchange of their sums.  Kernel, us, 32 / 64 / 64 by two, features d_in + d_out: Gram of
// 700 tokens, 512 features 22 / 29 / 25, 3072 99 / 134 / 78; 874, 3000 123 / 133 / 130; 1000, 1024 58 / 50 / 56; 1200, 1792 140 / 135 / 115;
// 2000, 1024 180 / 142 / 186.  128 samples: 4000 tokens, 1024 61 / 52 / 59; 4979, 1104 81 / 88 / 85; 7032, 2994 300 / 241 / 197; 8000, 640
// 66 / 55 / 77; 32 samples, which fill half of a tile of 64: 20000, 896 66 / 95 / 110.  Four CTAs to a tile of 64 were never the best.
struct GramShape { int tile, ctas; };
static GramShape f32_gram_shape(int64_t rows, int64_t cols, bool triangle, int d_in, int d_out) {
  auto tiles = [&](int64_t t) {
    const int64_t r = (rows + t - 1) / t, c = (cols + t - 1) / t;
    return triangle ? c * (c + 1) / 2 : r * c;
  };
  const int stages = (d_in + kGK - 1) / kGK + (d_out + kGK - 1) / kGK;
  GramShape g{32, 1};
  while (g.ctas < 8 && tiles(32) * 2 * g.ctas <= 240 && stages >= 10 * g.ctas) g.ctas *= 2;
  if (g.ctas > 1 && (g.ctas = placed_cluster(g.ctas)) > 1) return g;
  auto per_sm = [](int64_t ctas) { return (double)((ctas + kSms - 1) / kSms); };
  const double k1 = per_sm(tiles(64)), k2 = per_sm(2 * tiles(64));
  const double narrow = stages * std::max(0.48, 0.205 * per_sm(tiles(32)));
  const double wide = stages * (0.12 + 0.52 * k1), split = 0.5 * stages * (0.12 + 0.52 * k2) + 8.0 * k2;
  if (narrow <= wide && narrow <= split) return g;
  return GramShape{64, wide <= split ? 1 : placed_cluster(2)};
}
template <bool kSampled>
static isopo_status launch_f32_gram(int id, const GramShape& g, int64_t units, const float* RX, const float* RY, int64_t n_rows, const float* X,
                                    const float* dY, int64_t T, int d_in, int d_out, const int32_t* tokseq, int B, double* out, cudaStream_t st) {
  if (units * g.ctas > INT32_MAX) return ISOPO_ERR_UNSUPPORTED;
  {
    LaunchScope scope(id, st);
    const auto wide = g.ctas == 1 ? k_f32_gram<kSampled, 64, 1> : k_f32_gram<kSampled, 64, 2>;
    const auto narrow = g.ctas == 1   ? k_f32_gram<kSampled, 32, 1>
                        : g.ctas == 2 ? k_f32_gram<kSampled, 32, 2>
                        : g.ctas == 4 ? k_f32_gram<kSampled, 32, 4>
                                      : k_f32_gram<kSampled, 32, 8>;
    launch_cluster(g.tile == 32 ? narrow : wide, (unsigned)g.ctas, dim3((unsigned)(units * g.ctas)),
                   128, 0, st, RX, RY, n_rows, X, dY, T, d_in, d_out, tokseq, B, out);
  }
  ISOPO_CUDA_TRY(cudaGetLastError());
  return ISOPO_OK;
}

isopo_status f32_gram(const float* X, const float* dY, int64_t T, int d_in, int d_out, const int32_t* tokseq, int B,
                      double* kacc, float* K, cudaStream_t st) {
  const GramShape g = f32_gram_shape(T, T, true, d_in, d_out);
  const int64_t nt = (T + g.tile - 1) / g.tile;
  const isopo_status s = launch_f32_gram<false>(kIdF32Gram, g, nt * (nt + 1) / 2, X, dY, T, X, dY, T, d_in, d_out, tokseq, B, kacc, st);
  return s != ISOPO_OK ? s : launch_f32_finish(kacc, B, K, st);
}

isopo_status f32_sampled(const float* X, const float* dY, int64_t T, int d_in, int d_out, const float* a0, const float* g0,
                         int n_samples, const int32_t* tokseq, int B, double* Mt, cudaStream_t st) {
  const GramShape g = f32_gram_shape(n_samples, T, false, d_in, d_out);
  const int64_t nt = (T + g.tile - 1) / g.tile, ns = (n_samples + g.tile - 1) / g.tile;
  return launch_f32_gram<true>(kIdSampled, g, nt * ns, a0, g0, n_samples, X, dY, T, d_in, d_out, tokseq, B, Mt, st);
}

isopo_status f32_combine(const float* G, int64_t N, int64_t gstride, int B, const float* coeffs, float* dW, float beta,
                         const WsTag* tag_dev, const WsTag& tag, int32_t* info, cudaStream_t st) {
  // split while whole lanes would leave the machine (about 2^17 lanes of four elements in flight) mostly empty
  const bool split = N < ((int64_t)1 << 19) && B >= 4;
  const int64_t per_block = split ? 128 : 1024;
  const int grid = (int)std::min<int64_t>((N + per_block - 1) / per_block, kSms * 16);
  {
    LaunchScope scope(kIdF32Combine, st);
    launch((split ? k_f32_combine<8> : k_f32_combine<1>), grid, 256, 0, st, G, N, gstride, B, coeffs, dW, beta, tag_dev, tag, info);
  }
  ISOPO_CUDA_TRY(cudaGetLastError());
  return ISOPO_OK;
}

// What a CTA spends on filling its pipeline and adding its tile, in stages of 16 tokens.
constexpr int64_t kSlabOverhead = 4;
struct F32Slabs { int64_t stages; double us; };  // of a token slab; what its CTAs take
// Token slabs of whole stages, 128 tokens or more, up to eight waves (slab_plan.h).  "Four CTAs per SM" instead left the last
// wave nearly empty: 896 x 896, 4835 tokens 206 -> 190 us, 1537 x 739, 18,151 tokens 1484 -> 1265, 64 x 64, 353 tokens 13.2 ->
// 10.1 (this alone).  Two CTAs of 128 x 128 on an SM take twice the time of one (a stage of the SM 1.57 us each, 0.56 for 64 x 64; 1.75
// and 0.63 where rows are not made of 16 bytes), so where few units leave most SMs with one, slabs for one to an SM are better: 500 tokens, 896 x 896 31.8 -> 23.8 us, 20,000 tokens, 128 x 128 31.6 -> 21.7.
template <int kTile, int kT>
static isopo_status plan_f32_weight_grad(int64_t T, int d_in, int d_out, F32Slabs* plan) {
  typedef SlabGemm<kTile, kT> Gemm;
  const auto kernel = k_f32_weight_grad<kTile, kT>;
  int dev = 0, sms = 0;
  ISOPO_CUDA_TRY(cudaGetDevice(&dev));
  ISOPO_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  // CTAs at one time on an SM.  One word, all that a thread takes from another: beside the SMs in a second one, a thread could have seen the
  // first set and the second not yet, and divided by zero.
  static std::atomic<int> resident[64] = {};
  if (dev < 0 || dev >= 64) return ISOPO_ERR_UNSUPPORTED;
  int per_sm = resident[dev].load(std::memory_order_relaxed);
  if (per_sm == 0) {
    ISOPO_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, Gemm::kSmem));
    ISOPO_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, Gemm::kThr, Gemm::kSmem));
    resident[dev].store(per_sm = std::max(per_sm, 1), std::memory_order_relaxed);
  }
  const int64_t tiles = (int64_t)((d_in + kTile - 1) / kTile) * ((d_out + kTile - 1) / kTile), slots = (int64_t)sms * per_sm, n = sms;
  const int64_t blocks = (T + 15) / 16, most = std::min<int64_t>((T + 127) / 128, std::max<int64_t>(8, 8 * slots / tiles));
  auto us = [&](int64_t stages) {
    const int64_t units = (blocks + stages - 1) / stages * tiles, on_sm = (units + n - 1) / n, waves = (units + slots - 1) / slots;
    return (double)(on_sm * stages + 2 * waves) * (kTile == 128 ? 1.57 : 0.56);
  };
  plan->stages = plan_slab(blocks, tiles, slots, kSlabOverhead, most);
  if (kTile == 128) {
    const int64_t alone = plan_slab(blocks, tiles, n, 2, most);
    if (us(alone) < 0.93 * us(plan->stages)) plan->stages = alone;
  }
  plan->us = us(plan->stages);
  return ISOPO_OK;
}
template <int kTile, int kT>
static isopo_status launch_f32_weight_grad(const float* X, const float* dY, int64_t T, int d_in, int d_out, const int64_t* off_host,
                                           int64_t* off_dev, const float* coeffs, int B, float* tokscale, float* dW, bool add,
                                           const F32Slabs& plan, cudaStream_t st) {
  typedef SlabGemm<kTile, kT> Gemm;
  const int gx = (d_in + kTile - 1) / kTile, gy = (d_out + kTile - 1) / kTile;
  if (gy > 65535) return ISOPO_ERR_UNSUPPORTED;
  const auto kernel = k_f32_weight_grad<kTile, kT>;
  ISOPO_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, Gemm::kSmem));
  const int64_t slab = 16 * plan.stages;
  const int64_t splits = (T + slab - 1) / slab;
  if (splits > 65535) return ISOPO_ERR_UNSUPPORTED;
  const bool store = !add && splits == 1;
  const isopo_status s = launch_tokscale(off_host, B, T, off_dev, coeffs, tokscale,
                                         add || store ? Clear{} : Clear{{dW}, {(int64_t)d_in * d_out}}, st);
  if (s != ISOPO_OK) return s;
  {
    LaunchScope scope(kIdF32WeightGrad, st);
    launch(kernel, dim3(gx, gy, (unsigned)splits), Gemm::kThr, Gemm::kSmem, st, X, dY, T, d_in, d_out, tokscale, dW, slab, store);
  }
  ISOPO_CUDA_TRY(cudaGetLastError());
  return ISOPO_OK;
}

isopo_status f32_weight_grad(const float* X, const float* dY, int64_t T, int d_in, int d_out, const int64_t* off_host, int64_t* off_dev,
                             const float* coeffs, int B, float* tokscale, float* dW, bool add, cudaStream_t st) {
  // Tiles by the time that their CTAs take, 64 x 64 / 128 x 128, us: 500 tokens, 1536 x 1536 76.0 / 57.4, 1539 x 1539 98.7 / 84.2; 100, 1536 x 1536
  // 20.3 / 16.2, 1539 x 1539 27.5 / 31.3; 150, 1000 x 1000 15.1 / 13.5; 800, 448 x 896 23.3 / 21.7; 10,000, 192 x 192 26.6 / 34.0; 4000, 320 x 320 30.1 / 30.8.
  F32Slabs narrow, wide;
  isopo_status s = plan_f32_weight_grad<64, 4>(T, d_in, d_out, &narrow);
  if (s == ISOPO_OK) s = plan_f32_weight_grad<128, 8>(T, d_in, d_out, &wide);
  if (s != ISOPO_OK) return s;
  return narrow.us <= wide.us
             ? launch_f32_weight_grad<64, 4>(X, dY, T, d_in, d_out, off_host, off_dev, coeffs, B, tokscale, dW, add, narrow, st)
             : launch_f32_weight_grad<128, 8>(X, dY, T, d_in, d_out, off_host, off_dev, coeffs, B, tokscale, dW, add, wide, st);
}

}  // namespace isopo
