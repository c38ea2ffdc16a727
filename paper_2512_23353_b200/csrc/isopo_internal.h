// Internal declarations shared by the translation units of libisopo (not part of the C ABI).
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "isopo.h"

namespace isopo {

// Tile of the stored per-sequence gradients on the bf16 path: one tensor-core accumulator tile.
constexpr int kTileM = 128;  // rows of G (d_out)
constexpr int kTileN = 256;  // columns of G (d_in)

// Kernel identifiers: written to *info together with ISOPO_INFO_TIMEOUT, and the index of the
// per-kernel timing slots of isopo_profile_collect.
enum KernelId : int {
  kIdPrep = 0,
  kIdSeqGrad = 1,
  kIdNtk = 2,
  kIdGram = 3,
  kIdWeightGrad = 4,
  kIdCombine = 5,
  kIdTransform = 6,
  kIdMirror = 7,
  kIdF32SeqGrad = 8,
  kIdF32Ntk = 9,
  kIdF32Gram = 10,
  kIdF32WeightGrad = 11,
  kIdF32Combine = 12,
  kIdSampled = 13,     // M^T of the token-sampled estimator (tensor-core or float32 kernel)
  kIdSampledAux = 14,  // its gather and finishing kernels
  kIdScaleRows = 15,   // per-token scale of the narrower operand before the 2-CTA weight-gradient GEMM
  kIdWaitProbe = 16,   // isopo_selftest_bounded_wait
  kIdCount = 17
};

// Debug build (-DISOPO_DEBUG, libisopo_debug.so): every index a kernel computes for a global load, store or
// atomic of its own buffers (stored gradients, K, M^T, dW, the staged sequence tables) is compared with the
// buffer's extent first; an index outside it skips the access and records ISOPO_INFO_BOUNDS | kernel id in
// *info.  It stands in for a memory checker on the data-dependent addressing: ragged tails, the
// piece-blocked store, segment sums.  In the normal build the checks compile to nothing.
#ifdef ISOPO_DEBUG
__device__ __forceinline__ bool dbg_in_range(long long idx, long long n, int32_t* info, int id) {
  if (idx >= 0 && idx < n) return true;
  atomicCAS(info, 0, ISOPO_INFO_BOUNDS | id);
  return false;
}
#define ISOPO_IN_RANGE(idx, n, info, id) (::isopo::dbg_in_range((long long)(idx), (long long)(n), (info), (id)))
#else
#define ISOPO_IN_RANGE(idx, n, info, id) (true)
#endif

// Brackets one kernel launch with CUDA events while profiling is enabled (isopo_profile_enable);
// otherwise only counts the launch.
class LaunchScope {
 public:
  LaunchScope(int id, cudaStream_t st);
  ~LaunchScope();

 private:
  int slot_;
  cudaStream_t st_;
};

// Suspends event timing for the lifetime of the object (launch counting continues).
class ProfilingPause {
 public:
  ProfilingPause();
  ~ProfilingPause();

 private:
  bool was_on_;
};

// What isopo_layer_gram(MATERIALISE) leaves at the head of the workspace so that isopo_weight_grad can tell
// whether the stored gradients it is about to sum belong to the layer and microbatch it was called for.
struct WsTag {
  int64_t v[8];  // magic, dtype, T, d_in, d_out, B, hash of the offsets, 0
};
WsTag make_ws_tag(isopo_dtype dtype, int64_t T, int d_in, int d_out, int B, const int64_t* off_host);

// What lies at the head of a workspace on the materialised route.
struct WsHead {
  WsTag tag;
  uint32_t done;  // CTAs of the K pass that have added their share (bf16)
};

// What the bf16 gradient kernel takes as arguments besides its matrices, so that no launch of its own prepares it: the
// token offsets, the sequences longest first, and per projection the head to leave in its workspace and what the K pass behind it
// adds into, to be cleared.
struct StoredIntake {
  int32_t off[257];
  uint8_t order[256];
  int n_proj;
  WsTag tag[3];
  WsHead* head[3];
  float* acc[3];
  int n_acc;
};
void make_stored_intake(StoredIntake* a, const int64_t* off_host, int B, int n_proj, const WsTag* tag, WsHead* const* head,
                        float* const* acc, int n_acc);
// Extents of the sequences in working order to shared memory (`raw`: scratch there, kIntakeRawBytes).  Arguments are no
// memory of any predecessor's, so this may run before the wait for them.  The arguments are read as ordinary memory, a word
// per thread: indexing them directly goes through the constant cache, one word at a time (2.5 us at 236 sequences).
constexpr int kIntakeRawBytes = 257 * 4 + 256;
__device__ __forceinline__ void stored_extents(const StoredIntake& a, int B, int32_t* raw, int64_t* s_first, int* s_len, int* s_seq) {
  static_assert(offsetof(StoredIntake, order) == 257 * 4, "one run of words");
  const int32_t* src = a.off;
  asm volatile("" : "+l"(src));  // an address like any other
  for (int k = threadIdx.x; k < kIntakeRawBytes / 4; k += blockDim.x) raw[k] = src[k];
  __syncthreads();
  const uint8_t* order = reinterpret_cast<const uint8_t*>(raw + 257);
  for (int k = threadIdx.x; k < B; k += blockDim.x) {
    const int i = order[k], t0 = raw[i];
    s_first[k] = t0;
    s_len[k] = raw[i + 1] - t0;
    s_seq[k] = i;
  }
}
// The grid's share of the clearing; CTA 0 leaves the heads.
__device__ __forceinline__ void stored_heads(const StoredIntake& a) {
  for (int h = 0; h < a.n_proj; ++h) {
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < a.n_acc; e += gridDim.x * blockDim.x) a.acc[h][e] = 0.f;
    if (blockIdx.x == 0) {
      if (threadIdx.x < 8) a.head[h]->tag.v[threadIdx.x] = a.tag[h].v[threadIdx.x];
      if (threadIdx.x == 8) a.head[h]->done = 0u;
    }
  }
}

// How the bf16 stored route keeps G_i.  Split (isopo_set_store_format(ISOPO_STORE_E4M3_SPLIT)): two e4m3 planes of
// one byte per element each - `hi` = round(s_i G_i), `lo` = round(16 (s_i G_i - hi)) with a power-of-two scale s_i per
// sequence - in the same piece order.  The K pass reads only `hi` (half the bytes, kind::f8f6f4 MMAs) and takes the
// diagonal from `kdiag`, which the gradient GEMM sums in float32 from its accumulators; the combine reads both planes.
struct StoreFmt {
  int split;             // 0: bf16 (2 bytes per element), 1: e4m3 hi / lo planes
  const float* scales;   // [B] s_i
  float* kdiag;          // [B] sum of squares of G_i
};

struct WsLayout {
  size_t off_tag;      // WsHead (materialised path)
  size_t off_aux;      // float scales[B] | float kdiag[B]  (bf16 materialised path, split store)
  size_t off_offsets;  // int64 [B+1]
  size_t off_tokseq;   // int32 [T]: token -> sequence; the bf16 weight-gradient GEMM keeps float32 per-token scales here
  size_t off_kacc;     // float32 path: float64 [B*B] K accumulators (Gram), uint32 CTAs of the K pass that are done (materialised)
  size_t off_scaled;   // bf16 Gram path: copies of the operands at a pitch of whole lines (repitch_bytes), later the pre-scaled operand of the
                       // weight-gradient GEMM, bf16 [T, scaled_ld]
  size_t off_G;        // stored gradients (materialised path only)
  size_t off_kpart;    // per-CTA partial K (materialised path; bf16: in deterministic mode only)
  size_t off_ksums;    // bf16 materialised path above 32 sequences: what the K pass adds into, float [B][ntk_pitch(B)]; where the token map
                       // is when it has the room; 0: none, added into K itself
  size_t total;
  int scaled_ld;         // of the pre-scaled operand: line_pitch(min(d_in, d_out)), or the width itself in a workspace without that room
  int tiles_m, tiles_n;  // bf16 materialised layout: tiles per gradient
  int64_t n_pad;         // elements per stored gradient (row stride of G_flat)
};

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// In a workspace of `have` bytes: the areas that only make the kernels faster are left out, or hold fewer copies, where they do not fit
// (layout.total is then at most `have`, or what the others need), so that a workspace of 2 T min(d_in, d_out) bytes of scaled operand, or
// with no sums of the K pass, still serves.
WsLayout ws_layout(isopo_dtype dtype, int64_t T, int d_in, int d_out, int B, isopo_path resolved, size_t have = SIZE_MAX);

// Workspace of isopo_sampled_coefficients: the Gram-route prefix (offsets, token map), then
// the gathered rows a0 / g0, M^T and the denominator.
struct SampledLayout {
  size_t off_a0, off_g0, off_mt, off_den, total;
  int lda, ldg;  // of the sample rows: bf16 whole lines, in a workspace of `have` bytes that has the room
};
SampledLayout sampled_layout(isopo_dtype dtype, int64_t T, int d_in, int d_out, int B, int n_samples, size_t have = SIZE_MAX);

void set_cuda_error(cudaError_t e, const char* where);
#define ISOPO_CUDA_TRY(expr)                                  \
  do {                                                        \
    cudaError_t e__ = (expr);                                 \
    if (e__ != cudaSuccess) {                                 \
      ::isopo::set_cuda_error(e__, #expr);                    \
      return ISOPO_ERR_CUDA;                                  \
    }                                                         \
  } while (0)

// ---- programmatic dependent launch ----
// A layer is a chain of five to ten dependent kernels, several of them a few microseconds long.  The kernels of the
// library are launched so that their CTAs may be set up as soon as their predecessor in the stream lets them (not
// k_transform_large, launched with a cluster size alone, and the self-test's k_wait_probe), and wait for everything before
// them to be complete and visible before they touch memory: k_spectral, which runs beside its predecessor, before it ends.
// All CTAs of a kernel wait, so that the chain stays ordered end to end.  Work of other origin in the stream is ordered as always.
//   pdl_begin  waits, then lets the successor in while this kernel runs: kernels of one CTA per SM, which leave no room
//              beside them, and kernels of a few CTAs
//   pdl_wait   waits; the successor is let in when the last CTA leaves.  Kernels of several CTAs per SM: a successor let
//              in earlier finds a few SMs with room and is crowded onto them (a float32 layer of 102 sequences, 789
//              tokens: 184 us a pass when every kernel let its successor in at once, 133 us so)
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_begin() {
  pdl_wait();
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
// The kernel must call pdl_begin() or pdl_wait().  Errors are picked up by the cudaGetLastError() that follows every launch.
template <typename... Params, typename... Args>
inline void launch(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
}

// The same in clusters of `cluster` CTAs.
template <typename... Params, typename... Args>
inline void launch_cluster(void (*kernel)(Params...), unsigned cluster, dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = cluster;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
}

// The largest cluster of up to `wanted` (8, 4, 2 or 1) CTAs, each with an SM to itself, that the current context can place: where it has a
// part of a device, SMs of one group may be too few for it.  Asked at every call, as contexts of a device differ (0.2 us, where a kernel
// in clusters of more than one is to be launched).
int placed_cluster(int wanted);

// ---- launchers (each enqueues on `st` and returns a status; none synchronises) ----

// Up to three float32 regions that a launch clears for the kernels behind it (n = 0: none).
struct Clear {
  float* p[3];
  int64_t n[3];
};
// Clears the regions that the kernels behind this one add into (in place of a memset for each).
__device__ __forceinline__ void clear_regions(const Clear& c) {
  const int64_t first = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    if (c.n[k] == 0) continue;
    const int64_t quads = (reinterpret_cast<uintptr_t>(c.p[k]) & 15) == 0 ? c.n[k] / 4 : 0;
    for (int64_t e = first; e < quads; e += step) reinterpret_cast<float4*>(c.p[k])[e] = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int64_t e = 4 * quads + first; e < c.n[k]; e += step) c.p[k][e] = 0.f;
  }
}
// Row pitch of the library's own copies of bf16 operands, in elements: whole 128-byte lines.  TMA copies 128 bytes of a row at a time;
// where rows start anywhere, that is two lines of the L2 each: sampled estimator of 37,888 tokens, 128 samples, 2136 x 968 61 us, 2048 x
// 1024 39 us.
__host__ __device__ inline int line_pitch(int d) { return (d + 63) & ~63; }
// Rows that a launch copies to a pitch of whole lines for the kernels behind it (n operands).
constexpr int kMaxRepitch = 4;
struct Repitch {
  const uint4* src[kMaxRepitch];
  uint4* dst[kMaxRepitch];
  int d8[kMaxRepitch], p8[kMaxRepitch];  // row and pitch in 16-byte pieces
  int n;
};
// Token offsets as kernel arguments (no host-to-device copy); they are below 2^31 and travel as 32-bit values.
constexpr int kArgChunk = 384;   // the usual case; 1.5 KB of arguments
constexpr int kArgLarge = 2048;  // 8 KB
template <int kN> struct OffsetArgs { int32_t v[kN]; };
// The arguments as ordinary memory, a word per thread: indexed directly they go through the constant cache, one word at a time.
template <int kN>
__device__ __forceinline__ const int32_t* offsets_memory(const OffsetArgs<kN>& a) {
  const int32_t* from = a.v;
  asm volatile("" : "+l"(from));
  return from;
}
template <int kN>
inline void fill_offsets(OffsetArgs<kN>* a, const int64_t* off_host, int n) {
  for (int t = 0; t < n; ++t) a->v[t] = (int32_t)off_host[t];
}
// offsets and the token -> sequence map to the device, `clear` cleared
isopo_status launch_prep(const int64_t* off_host, int B, int64_t T, int64_t* off_dev, int32_t* tokseq, const Clear& clear,
                         cudaStream_t st);
// the same (fewer than kArgLarge sequences), and rows copied to another pitch
isopo_status launch_prep_repitch(const int64_t* off_host, int B, int64_t T, int64_t* off_dev, int32_t* tokseq, const Clear& clear,
                                 const Repitch& repitch, cudaStream_t st);
// the offsets alone
isopo_status launch_offsets(const int64_t* off_host, int B, int64_t* off_dev, const Clear& clear, cudaStream_t st);
// offsets and tokscale[t] = coeffs[sequence of token t] (float32 [T])
isopo_status launch_tokscale(const int64_t* off_host, int B, int64_t T, int64_t* off_dev, const float* coeffs,
                             float* tokscale, const Clear& clear, cudaStream_t st);
// true when every word of the tag in the workspace equals `want`; otherwise the first thread of the grid
// records ISOPO_INFO_STALE_WORKSPACE (device code, used by the combine kernels)
__device__ __forceinline__ bool ws_tag_matches(const WsTag* __restrict__ have, const WsTag& want, int32_t* info) {
  bool ok = true;
#pragma unroll
  for (int k = 0; k < 8; ++k) ok = ok && have->v[k] == want.v[k];
  if (!ok && blockIdx.x == 0 && threadIdx.x == 0) atomicCAS(info, 0, ISOPO_INFO_STALE_WORKSPACE);
  return ok;
}

// float32 path.  gstride: floats between the stored gradients of two sequences (WsLayout::n_pad, a multiple of 4)
// f32_seq_grad also leaves the tag and clears `done`, which f32_ntk counts in
isopo_status f32_seq_grad(const float* X, const float* dY, int d_in, int d_out, const int64_t* off_host, int64_t* off_dev,
                          int B, float* G, int64_t gstride, uint32_t* done, const WsTag& tag, WsTag* tag_dev, cudaStream_t st);
// part: f32_ntk_part_bytes of scratch
size_t f32_ntk_part_bytes(int64_t gstride, int B);
isopo_status f32_ntk(const float* G, int64_t gstride, int B, double* part, uint32_t* done, float* K, cudaStream_t st);
// M^T [n_samples, B] += of the sampled rows a0, g0
isopo_status f32_sampled(const float* X, const float* dY, int64_t T, int d_in, int d_out, const float* a0, const float* g0,
                         int n_samples, const int32_t* tokseq, int B, double* Mt, cudaStream_t st);
isopo_status f32_gram(const float* X, const float* dY, int64_t T, int d_in, int d_out, const int32_t* tokseq, int B,
                      double* kacc, float* K, cudaStream_t st);
isopo_status f32_combine(const float* G, int64_t N, int64_t gstride, int B, const float* coeffs, float* dW, float beta,
                         const WsTag* tag_dev, const WsTag& tag, int32_t* info, cudaStream_t st);
// as the bf16 ones below: prepares the tokens' scales and clears dW where it has to
isopo_status f32_weight_grad(const float* X, const float* dY, int64_t T, int d_in, int d_out, const int64_t* off_host, int64_t* off_dev,
                             const float* coeffs, int B, float* tokscale, float* dW, bool add, cudaStream_t st);

// bf16 tcgen05 path
isopo_status bf16_seq_grad(const void* X, const void* dY, int64_t T, int d_in, int d_out, const StoredIntake& in, int B,
                           const WsLayout& L, void* G, const StoreFmt& fmt, int32_t* info, cudaStream_t st);
// whether a layer of this shape keeps its gradients in the split e4m3 format under the current settings
bool use_split_store(const WsLayout& L, int B);
StoreFmt store_fmt(const WsLayout& L, int B, void* ws);
// s_i of every sequence from a sample of its token rows, kdiag = 0 (split store)
isopo_status launch_seq_scales(const void* X, const void* dY, int d_in, int d_out, const int64_t* off_dev, int B, float* scales,
                               float* kdiag, cudaStream_t st);
// the same for up to three projections that read one X, in one launch (L, dY, d_out, G: one entry per projection)
isopo_status bf16_seq_grad_pair_shared(const void* X, int n_proj, const void* const* dY, const int* d_out, int64_t T, int d_in,
                                       const StoredIntake& in, int B, const WsLayout* L, void* const* G, const StoreFmt* fmt,
                                       int32_t* info, cudaStream_t st);
// kpart != NULL (deterministic mode): every CTA of the K pass stores its partial triangle there ([kNtkMaxPartials][B * B] floats) and
// a second kernel sums them in order.  Otherwise they add one triangle into K, or by_boxes into rows of ntk_pitch(B) floats (`acc`); either
// has been cleared on this stream, and the last CTA or a second kernel completes K.
constexpr int kNtkMaxPartials = 160;
constexpr int kNtkSmemSums = 32;  // sequences up to which a CTA adds its groups of pieces in shared memory and then into K
inline int ntk_pitch(int B) { return (B + 3) & ~3; }
struct NtkPlan {
  int box_rows, ppb;  // rows of a piece inside a box, pieces per box
  long long nkb;      // boxes
  int grid, n_active;
  bool by_boxes, by_last;
};
isopo_status plan_ntk(const WsLayout& L, int B, bool split, bool deterministic, NtkPlan* plan);
isopo_status bf16_ntk(const NtkPlan& plan, const void* G, const WsLayout& L, int B, float* K, float* acc, WsHead* head, float* kpart,
                      const StoreFmt& fmt, int32_t* info, cudaStream_t st);
bool deterministic_mode();
// K[i][j] = K[j][i] for j < i (the Gram kernels fill the upper triangle)
isopo_status mirror_upper(float* K, int B, cudaStream_t st);
isopo_status bf16_combine(const void* G, const WsLayout& L, int d_in, int d_out, int B, const float* coeffs, float* dW,
                          float beta, const WsTag* tag_dev, const WsTag& tag, const StoreFmt& fmt, int32_t* info,
                          cudaStream_t st);
// The Gram and sampled kernels ADD into K and M^T: the caller has cleared them on this stream.
// (ld: elements from row to row)
isopo_status bf16_gram(const void* X, int ldx, const void* dY, int ldy, int64_t T, int d_in, int d_out, const int32_t* tokseq, int B,
                       float* K, int32_t* info, cudaStream_t st);
// 2-CTA tiles, one projection or several that share X: where they pay
bool bf16_gram_pair_pays(int64_t T, int d_in, const int* d_out, int n_heads, int sms);
isopo_status bf16_gram_pair(const void* X, int ldx, const void* const* dY, const int* ldy, int64_t T, int d_in, const int* d_out, int n_heads,
                            const int32_t* tokseq, int B, float* const* K, int32_t* info, cudaStream_t st);
isopo_status bf16_gram_shared(const void* X, int ldx, const void* const* dY, const int* ldy, int64_t T, int d_in, const int* d_out, int n_heads,
                              const int32_t* tokseq, int B, float* const* K, int32_t* info, cudaStream_t st);
// few tiles: a cluster of `ctas` CTAs shares the features of a tile (1: the kernels above are the better)
int gram_split_ctas(long long units, int d_in, int d_out, int sms);  // asks placed_cluster
isopo_status bf16_gram_split(int ctas, const void* X, int ldx, const void* const* dY, const int* ldy, int64_t T, int d_in, const int* d_out, int n_heads,
                             const int32_t* tokseq, int B, float* const* K, bool complete, int32_t* info, cudaStream_t st);
isopo_status bf16_sampled_split(int ctas, const void* X, const void* dY, int64_t T, int d_in, int d_out, const int32_t* tokseq, int B,
                                const void* A0, int lda, const void* G0, int ldg, int n_samples, float* Mt, int32_t* info, cudaStream_t st);
// The stand-alone weight gradients prepare what they need (offsets through off_dev, a cleared dW where its shares are added up);
// `add`: dW is added to.
// 1-CTA tiles, operand rows scaled in shared memory by the scales per token that a launch ahead leaves in `tokscale`
isopo_status bf16_weight_grad(const void* X, const void* dY, int64_t T, int d_in, int d_out, const int64_t* off_host,
                              int64_t* off_dev, const float* coeffs, int B, float* tokscale, float* dW, bool add, int32_t* info,
                              cudaStream_t st);
bool bf16_weight_grad_uses_pairs(int64_t T, int d_in, int d_out, int B);

// dW with the per-sequence coefficient applied when a segment's accumulator is drained (no scaled operand copy)
bool bf16_weight_grad_fold_applies(int64_t T, int d_in, int d_out, int B);
isopo_status bf16_weight_grad_fold(const void* X, const void* dY, int64_t T, int d_in, int d_out, const int64_t* off_host,
                                   int64_t* off_dev, const float* coeffs, int B, float* dW, bool add, int32_t* info, cudaStream_t st);
// a scaled copy of the narrower operand, then a plain GEMM in 2-CTA tiles
// (the offsets travel with the scaling pass, through off_dev above 2047 sequences)
isopo_status bf16_weight_grad_pair(const void* X, const void* dY, int64_t T, int d_in, int d_out, const int64_t* off_host,
                                   int64_t* off_dev, const float* coeffs, int B, void* scaled, int scaled_ld, float* dW, bool add,
                                   int32_t* info, cudaStream_t st);
// plain GEMM in runs of stages per pair; modelled time in stages of 256 columns
struct PlainPlan {
  long long run, cost;
  bool clear;  // dW has to be cleared ahead of it
};
PlainPlan plan_weight_grad_plain(int64_t T, int d_in, int d_out, bool add, int pairs);
isopo_status bf16_weight_grad_plain(const void* X, int ldx, const void* dY, int ldy, int64_t T, int d_in, int d_out, const PlainPlan& plan, bool add,
                                    float* dW, int32_t* info, cudaStream_t st);

// token-sampled estimator of Algorithm 1
isopo_status bf16_sampled(const void* X, const void* dY, int64_t T, int d_in, int d_out, const int32_t* tokseq, int B,
                          const void* A0, int lda, const void* G0, int ldg, int n_samples, float* Mt, int32_t* info, cudaStream_t st);
isopo_status sampled_coefficients(const void* X, const void* dY, isopo_dtype dtype, int64_t T, int d_in, int d_out,
                                  const int32_t* tokseq, int B, const int64_t* rows_host, int n_samples, char* ws,
                                  const SampledLayout& S, const float* A, float lambda, float* coeffs, float* F2,
                                  int32_t* info, cudaStream_t st);

// transform (all variants)
size_t transform_large_workspace_bytes(int B);
isopo_status transform_large(const float* K, const float* A, int B, float lambda, float* coeffs, float* scratch,
                             int32_t* info, cudaStream_t st);
// the same without a cluster, any B whose diagonal blocks fit shared memory (ISOPO_MAX_LARGE_SEQS)
isopo_status transform_one_cta(const float* K, const float* A, int B, float lambda, float* coeffs, float* scratch, int32_t* info,
                               cudaStream_t st);
isopo_status transform(const float* K, const float* A, int B, isopo_variant v, float lambda, const float* pqr_regs_host,
                       const float* rel_state, float* coeffs, int32_t* info, cudaStream_t st);
isopo_status transform_batched(int n, const float* const* K, const float* A, int B, isopo_variant v, const float* lambda,
                               const float* pqr_regs_host, const float* const* rel_state, float* const* coeffs,
                               int32_t* info, cudaStream_t st);
size_t spectral_workspace_bytes();
isopo_status spectral(const float* K, const float* A, int B, float lambda, float rel_cutoff, float* coeffs, float* eig,
                      void* ws, int32_t* info, cudaStream_t st);
isopo_status spectral_batched(int n, const float* const* K, const float* A, int B, const float* lambda,
                              float rel_cutoff, float* const* coeffs, float* const* eig, void* ws, int32_t* info,
                              cudaStream_t st);
isopo_status wait_probe(long long limit_clocks, int32_t* info, int32_t* roles_at_teardown, cudaStream_t st);
isopo_status reg_ema_update(const float* K, int B, float decay, float* state, cudaStream_t st);

}  // namespace isopo
