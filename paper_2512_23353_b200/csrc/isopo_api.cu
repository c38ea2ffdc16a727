// C-ABI entry points of libisopo: argument validation, workspace layout, path choice, dispatch.
// Every step of the path runs in the CUDA kernels launched from here; there is no host arithmetic
// on the data and no CPU fallback.
#include <cstdio>
#include <cstring>
#include <algorithm>
#include <vector>

#include <nvtx3/nvToolsExt.h>

#include "isopo_internal.h"

namespace isopo {

// NVTX range named after the entry point, open for the duration of the host call (the kernels it
// enqueues appear under it in a profiler's timeline; without a profiler attached this is a no-op).
struct ApiRange {
  explicit ApiRange(const char* name) { nvtxRangePushA(name); }
  ~ApiRange() { nvtxRangePop(); }
};

static thread_local char g_cuda_err[256] = "no error";

void set_cuda_error(cudaError_t e, const char* where) {
  if (e == cudaSuccess)
    snprintf(g_cuda_err, sizeof(g_cuda_err), "%s", where);  // a plain explanation, no CUDA error behind it
  else
    snprintf(g_cuda_err, sizeof(g_cuda_err), "%s: %s (%s)", cudaGetErrorName(e), cudaGetErrorString(e), where);
}

static bool g_deterministic = false;
bool deterministic_mode() { return g_deterministic; }
static isopo_store_format g_store_format = ISOPO_STORE_BF16;

// The split store lives in the 2-CTA gradient GEMM and sums the diagonal of K with float atomics: layers that
// take the 1-CTA kernel, and everything in deterministic mode, keep the bf16 store.
bool use_split_store(const WsLayout& L, int B) {
  return g_store_format == ISOPO_STORE_E4M3_SPLIT && !g_deterministic && B <= 256 && (L.tiles_m % 2 == 0 || L.tiles_m >= 7);
}
StoreFmt store_fmt(const WsLayout& L, int B, void* ws) {
  float* aux = (float*)((char*)ws + L.off_aux);
  return StoreFmt{use_split_store(L, B) ? 1 : 0, aux, aux + B};
}

// ---- measurement hooks ----
struct ProfRecord { int id; cudaEvent_t a, b; };
static bool g_prof_on = false;
static std::vector<ProfRecord> g_prof;
static std::vector<cudaEvent_t> g_event_pool;
static int64_t g_launches[kIdCount] = {};

static cudaEvent_t take_event() {
  if (!g_event_pool.empty()) {
    cudaEvent_t e = g_event_pool.back();
    g_event_pool.pop_back();
    return e;
  }
  cudaEvent_t e = nullptr;
  cudaEventCreate(&e);
  return e;
}

LaunchScope::LaunchScope(int id, cudaStream_t st) : slot_(-1), st_(st) {
  ++g_launches[id];
  if (!g_prof_on) return;
  ProfRecord r{id, take_event(), take_event()};
  if (!r.a || !r.b) return;
  cudaEventRecord(r.a, st);
  slot_ = (int)g_prof.size();
  g_prof.push_back(r);
}

LaunchScope::~LaunchScope() {
  if (slot_ >= 0) cudaEventRecord(g_prof[slot_].b, st_);
}

ProfilingPause::ProfilingPause() : was_on_(g_prof_on) { g_prof_on = false; }
ProfilingPause::~ProfilingPause() { g_prof_on = was_on_; }

// Copies of the Gram route's operands at a pitch of whole lines, where theirs is none: from 1000 tokens on the token tiles' many reads of
// them outweigh a pass over the inputs.  isopo_layer_gram as they are / copied, us: 600 tokens, 2160 x 1032 15.1 / 16.6; 1000 19.0 / 17.8;
// 1919, 1080 x 312 17.6 / 14.8; 5000, 2136 x 968 70 / 64; 15,000, 1080 x 312 238 / 204; 40,000, 232 x 600 1184 / 885.
static bool repitch_pays(int64_t T, int B) { return T >= 1000 && B + 1 <= kArgLarge; }
static size_t repitch_bytes(int64_t T, int d) { return d % 64 ? align_up((size_t)2 * (size_t)T * (size_t)line_pitch(d), 1024) : 0; }
// What is asked for to hold them: X's and dY's, each unless it takes the two past 2 GiB.  (300,000 tokens of 8200 x 72, which need 0.04 GB
// without copies, asked for 5.0; now 0.08.)  They pay for lopsided layers too: in place / copied, 30,000 tokens, 8200 x 72 (0.5 GB) 8.4 /
// 6.5 ms, 1000 x 8200 9.6 / 7.1; 3000, 8200 x 72 148 / 94 us.
constexpr size_t kRepitchMost = (size_t)2 << 30;
static size_t repitch_room(int64_t T, int d_in, int d_out, int B) {
  if (!repitch_pays(T, B)) return 0;
  const size_t x = repitch_bytes(T, d_in), y = repitch_bytes(T, d_out), first = x <= kRepitchMost ? x : 0;
  return first + y <= kRepitchMost ? first + y : first;
}
struct GramOperands {
  const void* X;
  const void* dY[3];
  int ldx, ldy[3];
  Repitch repitch;
};
// What of X and the n dY has to be copied and has room there, X and the widest first.
static GramOperands gram_operands(const void* X, int d_in, int n, const void* const* dY, const int* d_out, int64_t T, int B, char* room,
                                  size_t bytes) {
  GramOperands g{};
  g.X = X;
  g.ldx = d_in;
  for (int h = 0; h < n; ++h) { g.dY[h] = dY[h]; g.ldy[h] = d_out[h]; }
  if (!repitch_pays(T, B)) return g;
  auto take = [&](const void** p, int* ld) {
    const size_t need = repitch_bytes(T, *ld);
    if (need == 0 || need > bytes) return;
    const int k = g.repitch.n++;
    g.repitch.src[k] = (const uint4*)*p;
    g.repitch.dst[k] = (uint4*)room;
    g.repitch.d8[k] = *ld / 8;
    g.repitch.p8[k] = line_pitch(*ld) / 8;
    *p = room;
    *ld = line_pitch(*ld);
    room += need;
    bytes -= need;
  };
  take(&g.X, &g.ldx);
  bool done[3] = {};
  for (int k = 0; k < n; ++k) {
    int widest = -1;
    for (int h = 0; h < n; ++h)
      if (!done[h] && (widest < 0 || d_out[h] > d_out[widest])) widest = h;
    done[widest] = true;
    take(&g.dY[widest], &g.ldy[widest]);
  }
  return g;
}

WsLayout ws_layout(isopo_dtype dtype, int64_t T, int d_in, int d_out, int B, isopo_path resolved, size_t have) {
  WsLayout L{};
  size_t p = 0;
  L.off_tag = p;
  p = align_up(p + sizeof(WsHead), 1024);
  L.off_aux = p;
  if (dtype == ISOPO_BF16 && resolved == ISOPO_PATH_MATERIALISE) p = align_up(p + 2 * sizeof(float) * (size_t)B, 1024);
  L.off_offsets = p;
  p = align_up(p + sizeof(int64_t) * (size_t)(B + 1), 1024);
  L.off_tokseq = p;
  p = align_up(p + sizeof(int32_t) * (size_t)T, 1024);
  L.off_kacc = p;
  if (dtype == ISOPO_F32)
    p = align_up(p + (resolved == ISOPO_PATH_MATERIALISE ? sizeof(uint32_t) : sizeof(double) * (size_t)B * (size_t)B), 1024);
  L.off_scaled = p;
  L.scaled_ld = std::min(d_in, d_out);
  if (dtype == ISOPO_BF16 && resolved == ISOPO_PATH_GRAM) {
    auto scaled = [&](int ld) { return align_up((size_t)2 * (size_t)T * (size_t)ld, 1024); };
    const size_t bare = scaled(L.scaled_ld), lines = scaled(line_pitch(L.scaled_ld));
    const size_t left = have < p + bare ? bare : (have - p) / 1024 * 1024;
    const size_t room = std::min(left, std::max(lines, repitch_room(T, d_in, d_out, B)));  // as much of it as there is
    if (room >= lines) L.scaled_ld = line_pitch(L.scaled_ld);
    p += room;
  }
  L.off_G = p;
  if (dtype == ISOPO_BF16) {
    L.tiles_m = (d_out + kTileM - 1) / kTileM;
    L.tiles_n = (d_in + kTileN - 1) / kTileN;
    L.n_pad = (int64_t)((d_out + 31) / 32 * 32) * d_in;  // pieces of 32 rows x 8 columns (tc_common.cuh)
    if (resolved == ISOPO_PATH_MATERIALISE) p = align_up(p + (size_t)2 * (size_t)B * (size_t)L.n_pad, 1024);
    L.off_kpart = p;
    if (resolved == ISOPO_PATH_MATERIALISE && deterministic_mode())
      p = align_up(p + sizeof(float) * (size_t)kNtkMaxPartials * (size_t)B * (size_t)B, 1024);
    else if (resolved == ISOPO_PATH_MATERIALISE && B > kNtkSmemSums) {
      const size_t bytes = sizeof(float) * (size_t)B * (size_t)ntk_pitch(B), full = align_up(p + bytes, 1024);
      if (bytes <= sizeof(int32_t) * (size_t)T) L.off_ksums = L.off_tokseq;
      else if (have >= full) { L.off_ksums = p; p = full; }
    }
  } else {
    L.tiles_m = L.tiles_n = 0;
    L.n_pad = ((int64_t)d_in * d_out + 3) / 4 * 4;
    if (resolved == ISOPO_PATH_MATERIALISE) p = align_up(p + (size_t)4 * (size_t)B * (size_t)L.n_pad, 1024);
    L.off_kpart = p;
    if (resolved == ISOPO_PATH_MATERIALISE) p = align_up(p + f32_ntk_part_bytes(L.n_pad, B), 1024);
  }
  L.total = p;
  return L;
}

WsTag make_ws_tag(isopo_dtype dtype, int64_t T, int d_in, int d_out, int B, const int64_t* off_host) {
  // four interleaved multiply-xorshift chains over the offsets, one word at a time (a byte at a time, each multiplication
  // waiting for the one before, took 2.5 us at 256 sequences)
  uint64_t lane[4] = {1469598103934665603ull, 0x9e3779b97f4a7c15ull, 0xc2b2ae3d27d4eb4full, 0x165667b19e3779f9ull};
  for (int i = 0; i <= B; ++i) {
    uint64_t& h = lane[i & 3];
    h = (h ^ (uint64_t)off_host[i]) * 0xff51afd7ed558ccdull;
    h ^= h >> 32;
  }
  uint64_t h = lane[0];
  for (int k = 1; k < 4; ++k) { h = (h ^ lane[k]) * 0xff51afd7ed558ccdull; h ^= h >> 32; }
  WsTag t{};
  t.v[0] = 0x49534f504f5f4753ll;
  t.v[1] = (int64_t)dtype; t.v[2] = T; t.v[3] = d_in; t.v[4] = d_out; t.v[5] = B; t.v[6] = (int64_t)h;
  if (dtype == ISOPO_BF16) {  // the format the stored gradients of this shape are kept in right now
    const WsLayout L = ws_layout(dtype, T, d_in, d_out, B, ISOPO_PATH_MATERIALISE);
    t.v[7] = use_split_store(L, B) ? 1 : 0;
  }
  return t;
}

static bool sizes_ok(isopo_dtype dtype, int64_t T, int d_in, int d_out, int B) {
  if (dtype != ISOPO_F32 && dtype != ISOPO_BF16) return false;
  if (T < 1 || B < 1 || d_in < 1 || d_out < 1 || (int64_t)B > T) return false;
  if (T > ((int64_t)1 << 31) - 1024) return false;  // token coordinates are 32-bit in the tensor maps
  return true;
}

static isopo_status check_layer_args(const void* X, const void* dY, isopo_dtype dtype, int64_t T, int d_in, int d_out,
                                     const int64_t* off, int B, isopo_path path, const void* ws) {
  if (!X || !dY || !off || !ws) return ISOPO_ERR_INVALID_ARG;
  if (!sizes_ok(dtype, T, d_in, d_out, B)) return ISOPO_ERR_INVALID_ARG;
  if (path != ISOPO_PATH_AUTO && path != ISOPO_PATH_GRAM && path != ISOPO_PATH_MATERIALISE)
    return ISOPO_ERR_INVALID_ARG;
  if (((uintptr_t)X & 15) || ((uintptr_t)dY & 15) || ((uintptr_t)ws & 1023)) return ISOPO_ERR_INVALID_ARG;
  if (off[0] != 0 || off[B] != T) return ISOPO_ERR_INVALID_ARG;
  for (int i = 0; i < B; ++i)
    if (off[i + 1] <= off[i]) return ISOPO_ERR_INVALID_ARG;
  if (dtype == ISOPO_BF16 && ((d_in & 7) || (d_out & 7))) return ISOPO_ERR_UNSUPPORTED;
  return ISOPO_OK;
}

static isopo_path resolve_path(isopo_dtype dtype, int64_t T, int d_in, int d_out, int B, isopo_path path) {
  return path == ISOPO_PATH_AUTO ? isopo_choose_path(dtype, T, d_in, d_out, B) : path;
}

}  // namespace isopo

using namespace isopo;

extern "C" {

const char* isopo_status_string(isopo_status s) {
  switch (s) {
    case ISOPO_OK: return "ISOPO_OK";
    case ISOPO_ERR_INVALID_ARG: return "ISOPO_ERR_INVALID_ARG";
    case ISOPO_ERR_UNSUPPORTED: return "ISOPO_ERR_UNSUPPORTED";
    case ISOPO_ERR_WORKSPACE: return "ISOPO_ERR_WORKSPACE";
    case ISOPO_ERR_CUDA: return "ISOPO_ERR_CUDA";
  }
  return "ISOPO_ERR_UNKNOWN";
}

const char* isopo_last_cuda_error(void) { return g_cuda_err; }

void isopo_profile_enable(int on) { g_prof_on = on != 0; }

void isopo_set_deterministic(int on) { g_deterministic = on != 0; }
isopo_status isopo_set_store_format(isopo_store_format f) {
  if (f != ISOPO_STORE_BF16 && f != ISOPO_STORE_E4M3_SPLIT) return ISOPO_ERR_INVALID_ARG;
  g_store_format = f;
  return ISOPO_OK;
}
isopo_store_format isopo_get_store_format(void) { return g_store_format; }
int isopo_get_deterministic(void) { return g_deterministic ? 1 : 0; }
int isopo_debug_build(void) {
#ifdef ISOPO_DEBUG
  return 1;
#else
  return 0;
#endif
}

isopo_status isopo_profile_collect(double* ms_by_kernel, int64_t* launches_by_kernel) {
  if (!ms_by_kernel || !launches_by_kernel) return ISOPO_ERR_INVALID_ARG;
  for (int k = 0; k < kIdCount; ++k) { ms_by_kernel[k] = 0.0; launches_by_kernel[k] = g_launches[k]; g_launches[k] = 0; }
  isopo_status rc = ISOPO_OK;
  for (const ProfRecord& r : g_prof) {
    float ms = 0.f;
    cudaError_t e = cudaEventSynchronize(r.b);
    if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, r.a, r.b);
    if (e != cudaSuccess) { set_cuda_error(e, "isopo_profile_collect"); rc = ISOPO_ERR_CUDA; }
    ms_by_kernel[r.id] += ms;
    g_event_pool.push_back(r.a);
    g_event_pool.push_back(r.b);
  }
  g_prof.clear();
  return rc;
}

const char* isopo_kernel_name(int id) {
  static const char* names[kIdCount] = {"k_tokseq", "k_bf16_seq_grad", "k_bf16_ntk", "k_bf16_gram", "k_bf16_weight_grad",
                                        "k_bf16_combine", "k_transform", "k_mirror_upper", "k_f32_seq_grad",
                                        "k_f32_ntk", "k_f32_gram", "k_f32_weight_grad", "k_f32_combine",
                                        "k_sampled", "k_sampled_aux", "k_scale_rows", "k_wait_probe"};
  return id >= 0 && id < kIdCount ? names[id] : "unknown";
}

isopo_path isopo_choose_path(isopo_dtype dtype, int64_t T, int d_in, int d_out, int B) {
  if (!sizes_ok(dtype, T, d_in, d_out, B)) return ISOPO_PATH_GRAM;
  if (dtype == ISOPO_BF16 && B > 256) return ISOPO_PATH_GRAM;  // stored-gradient kernels hold all B rows on chip
  // Modelled extra time over the plain dW GEMM (which both routes pay once).
  const double peak = dtype == ISOPO_BF16 ? 1.39e15 : 4.0e13;  // flop/s: tcgen05 bf16 vs SIMT fp32
  const double bw = 6.5e12;                                     // HBM bytes/s
  const double elt = dtype == ISOPO_BF16 ? 2.0 : 4.0;
  const double N = (double)d_in * (double)d_out;
  const double t_gram = (double)(d_in + d_out) * (double)T * (double)T / peak;
  const double t_mat = (double)B * (double)B * N / peak + 3.0 * elt * (double)B * N / bw;
  return t_gram < t_mat ? ISOPO_PATH_GRAM : ISOPO_PATH_MATERIALISE;
}

size_t isopo_workspace_bytes(isopo_dtype dtype, int64_t T, int d_in, int d_out, int B, isopo_path path) {
  if (!sizes_ok(dtype, T, d_in, d_out, B)) return 0;
  if (path != ISOPO_PATH_AUTO && path != ISOPO_PATH_GRAM && path != ISOPO_PATH_MATERIALISE) return 0;
  return ws_layout(dtype, T, d_in, d_out, B, resolve_path(dtype, T, d_in, d_out, B, path)).total;
}

isopo_status isopo_layer_gram(const void* X, const void* dY, isopo_dtype dtype, int64_t T, int d_in, int d_out,
                              const int64_t* seq_offsets_host, int B, isopo_path path, float* K, void* ws,
                              size_t ws_bytes, int32_t* info, void* cuda_stream) {
  ApiRange nvtx_range("isopo_layer_gram");
  if (!K || !info) return ISOPO_ERR_INVALID_ARG;
  isopo_status s = check_layer_args(X, dY, dtype, T, d_in, d_out, seq_offsets_host, B, path, ws);
  if (s != ISOPO_OK) return s;
  const isopo_path rp = resolve_path(dtype, T, d_in, d_out, B, path);
  if (dtype == ISOPO_BF16 && rp == ISOPO_PATH_MATERIALISE && B > 256) return ISOPO_ERR_UNSUPPORTED;
  const WsLayout L = ws_layout(dtype, T, d_in, d_out, B, rp, ws_bytes);
  if (ws_bytes < L.total) return ISOPO_ERR_WORKSPACE;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  char* w = (char*)ws;
  int64_t* off_dev = (int64_t*)(w + L.off_offsets);
  int32_t* tokseq = (int32_t*)(w + L.off_tokseq);
  WsTag* tag_dev = (WsTag*)(w + L.off_tag);
  if (dtype == ISOPO_BF16 && rp == ISOPO_PATH_MATERIALISE) {
    void* G = w + L.off_G;
    WsHead* head = (WsHead*)(w + L.off_tag);
    const WsTag tag = make_ws_tag(dtype, T, d_in, d_out, B, seq_offsets_host);
    StoredIntake in;
    const StoreFmt fmt = store_fmt(L, B, ws);
    NtkPlan plan;
    if ((s = plan_ntk(L, B, fmt.split, deterministic_mode(), &plan)) != ISOPO_OK) return s;
    float* acc = plan.by_boxes ? (float*)(w + L.off_ksums) : K;
    make_stored_intake(&in, seq_offsets_host, B, 1, &tag, &head, &acc, plan.by_boxes ? B * ntk_pitch(B) : B * B);
    if (fmt.split) {
      s = launch_offsets(seq_offsets_host, B, off_dev, Clear{}, st);
      if (s == ISOPO_OK) s = launch_seq_scales(X, dY, d_in, d_out, off_dev, B, (float*)fmt.scales, fmt.kdiag, st);
      if (s != ISOPO_OK) return s;
    }
    s = bf16_seq_grad(X, dY, T, d_in, d_out, in, B, L, G, fmt, info, st);
    if (s != ISOPO_OK) return s;
    return bf16_ntk(plan, G, L, B, K, acc, head, deterministic_mode() ? (float*)(w + L.off_kpart) : nullptr, fmt, info, st);
  }
  if (dtype == ISOPO_F32 && rp == ISOPO_PATH_MATERIALISE) {
    float* G = (float*)(w + L.off_G);
    uint32_t* done = (uint32_t*)(w + L.off_kacc);
    s = f32_seq_grad((const float*)X, (const float*)dY, d_in, d_out, seq_offsets_host, off_dev, B, G, L.n_pad, done,
                     make_ws_tag(dtype, T, d_in, d_out, B, seq_offsets_host), tag_dev, st);
    return s != ISOPO_OK ? s : f32_ntk(G, L.n_pad, B, (double*)(w + L.off_kpart), done, K, st);
  }
  double* kacc = (double*)(w + L.off_kacc);
  const int64_t bb = (int64_t)B * B;
  if (dtype == ISOPO_F32) {
    s = launch_prep(seq_offsets_host, B, T, off_dev, tokseq, Clear{{(float*)kacc}, {2 * bb}}, st);
    return s != ISOPO_OK ? s : f32_gram((const float*)X, (const float*)dY, T, d_in, d_out, tokseq, B, kacc, K, st);
  }
  const GramOperands g = gram_operands(X, d_in, 1, &dY, &d_out, T, B, w + L.off_scaled, L.off_G - L.off_scaled);
  s = g.repitch.n ? launch_prep_repitch(seq_offsets_host, B, T, off_dev, tokseq, Clear{{K}, {bb}}, g.repitch, st)
                  : launch_prep(seq_offsets_host, B, T, off_dev, tokseq, Clear{{K}, {bb}}, st);
  return s != ISOPO_OK ? s : bf16_gram(g.X, g.ldx, g.dY[0], g.ldy[0], T, d_in, d_out, tokseq, B, K, info, st);
}

isopo_status isopo_layer_gram_shared_x(const void* X, int n_proj, const void* const* dY, const int* d_out, isopo_dtype dtype,
                                       int64_t T, int d_in, const int64_t* seq_offsets_host, int B, float* const* K,
                                       void* ws, size_t ws_bytes, int32_t* info, void* cuda_stream) {
  ApiRange nvtx_range("isopo_layer_gram_shared_x");
  if (!dY || !d_out || !K || !info || n_proj < 1 || n_proj > 3) return ISOPO_ERR_INVALID_ARG;
  if (dtype != ISOPO_BF16) return ISOPO_ERR_UNSUPPORTED;
  int d_max = 0;
  for (int h = 0; h < n_proj; ++h) {
    if (!K[h]) return ISOPO_ERR_INVALID_ARG;
    isopo_status s = check_layer_args(X, dY[h], dtype, T, d_in, d_out[h], seq_offsets_host, B, ISOPO_PATH_GRAM, ws);
    if (s != ISOPO_OK) return s;
    d_max = std::max(d_max, d_out[h]);
  }
  const WsLayout L = ws_layout(dtype, T, d_in, d_max, B, ISOPO_PATH_GRAM, ws_bytes);
  if (ws_bytes < L.total) return ISOPO_ERR_WORKSPACE;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  char* w = (char*)ws;
  int32_t* tokseq = (int32_t*)(w + L.off_tokseq);
  Clear clear{};
  for (int h = 0; h < n_proj; ++h) { clear.p[h] = K[h]; clear.n[h] = (int64_t)B * B; }
  const GramOperands g = gram_operands(X, d_in, n_proj, dY, d_out, T, B, w + L.off_scaled, L.off_G - L.off_scaled);
  int64_t* off_dev = (int64_t*)(w + L.off_offsets);
  const isopo_status s = g.repitch.n ? launch_prep_repitch(seq_offsets_host, B, T, off_dev, tokseq, clear, g.repitch, st)
                                     : launch_prep(seq_offsets_host, B, T, off_dev, tokseq, clear, st);
  return s != ISOPO_OK ? s : bf16_gram_shared(g.X, g.ldx, g.dY, g.ldy, T, d_in, d_out, n_proj, tokseq, B, K, info, st);
}

isopo_status isopo_layer_gram_shared_x_stored(const void* X, int n_proj, const void* const* dY, const int* d_out,
                                              isopo_dtype dtype, int64_t T, int d_in, const int64_t* seq_offsets_host, int B,
                                              float* const* K, void* const* ws, const size_t* ws_bytes, int32_t* info,
                                              void* cuda_stream) {
  ApiRange nvtx_range("isopo_layer_gram_shared_x_stored");
  if (!dY || !d_out || !K || !ws || !ws_bytes || !info || n_proj < 1 || n_proj > 3) return ISOPO_ERR_INVALID_ARG;
  if (dtype != ISOPO_BF16 || B > 256) return ISOPO_ERR_UNSUPPORTED;
  WsLayout L[3];
  WsTag tag[3];
  int64_t* off_dev = nullptr;
  WsHead* head[3];
  void* G[3];
  float* acc[3];
  StoreFmt fmt[3];
  bool pairs_fit = true;
  for (int h = 0; h < n_proj; ++h) {
    if (!K[h]) return ISOPO_ERR_INVALID_ARG;
    isopo_status s = check_layer_args(X, dY[h], dtype, T, d_in, d_out[h], seq_offsets_host, B, ISOPO_PATH_MATERIALISE, ws[h]);
    if (s != ISOPO_OK) return s;
    for (int g = 0; g < h; ++g)
      if (ws[g] == ws[h]) return ISOPO_ERR_INVALID_ARG;  // every projection keeps its own gradients
    L[h] = ws_layout(dtype, T, d_in, d_out[h], B, ISOPO_PATH_MATERIALISE, ws_bytes[h]);
    if (ws_bytes[h] < L[h].total) return ISOPO_ERR_WORKSPACE;
    char* w = (char*)ws[h];
    tag[h] = make_ws_tag(dtype, T, d_in, d_out[h], B, seq_offsets_host);
    if (h == 0) off_dev = (int64_t*)(w + L[h].off_offsets);
    head[h] = (WsHead*)(w + L[h].off_tag);
    G[h] = w + L[h].off_G;
    fmt[h] = store_fmt(L[h], B, ws[h]);
    pairs_fit = pairs_fit && (L[h].tiles_m % 2 == 0 || L[h].tiles_m >= 7);
  }
  cudaStream_t st = (cudaStream_t)cuda_stream;
  isopo_status s = ISOPO_OK;
  bool have_offsets = false;
  for (int h = 0; h < n_proj; ++h)
    if (fmt[h].split) {
      if (!have_offsets) s = launch_offsets(seq_offsets_host, B, off_dev, Clear{}, st);
      have_offsets = true;
      if (s == ISOPO_OK) s = launch_seq_scales(X, dY[h], d_in, d_out[h], off_dev, B, (float*)fmt[h].scales, fmt[h].kdiag, st);
      if (s != ISOPO_OK) return s;
    }
  NtkPlan plan[3];  // by_boxes is the same for all: the number of sequences says, and whether all have the room
  for (int h = 0; h < n_proj; ++h)
    if (L[h].off_ksums == 0)
      for (int g = 0; g < n_proj; ++g) L[g].off_ksums = 0;
  for (int h = 0; h < n_proj; ++h) {
    if ((s = plan_ntk(L[h], B, fmt[h].split, deterministic_mode(), &plan[h])) != ISOPO_OK) return s;
    acc[h] = plan[h].by_boxes ? (float*)((char*)ws[h] + L[h].off_ksums) : K[h];
  }
  const int n_acc = plan[0].by_boxes ? B * ntk_pitch(B) : B * B;
  StoredIntake in;
  if (pairs_fit) {
    make_stored_intake(&in, seq_offsets_host, B, n_proj, tag, head, acc, n_acc);
    s = bf16_seq_grad_pair_shared(X, n_proj, dY, d_out, T, d_in, in, B, L, G, fmt, info, st);
    if (s != ISOPO_OK) return s;
  } else {  // a projection with an odd, small number of 128-row tiles would idle half of its pairs: one launch each
    for (int h = 0; h < n_proj; ++h) {
      make_stored_intake(&in, seq_offsets_host, B, 1, tag + h, head + h, acc + h, n_acc);
      s = bf16_seq_grad(X, dY[h], T, d_in, d_out[h], in, B, L[h], G[h], fmt[h], info, st);
      if (s != ISOPO_OK) return s;
    }
  }
  for (int h = 0; h < n_proj; ++h) {
    float* kpart = deterministic_mode() ? (float*)((char*)ws[h] + L[h].off_kpart) : nullptr;
    s = bf16_ntk(plan[h], G[h], L[h], B, K[h], acc[h], head[h], kpart, fmt[h], info, st);
    if (s != ISOPO_OK) return s;
  }
  return ISOPO_OK;
}

size_t isopo_sampled_workspace_bytes(isopo_dtype dtype, int64_t T, int d_in, int d_out, int B, int n_samples) {
  if (!sizes_ok(dtype, T, d_in, d_out, B) || n_samples < 1 || n_samples > ISOPO_MAX_SAMPLES) return 0;
  return sampled_layout(dtype, T, d_in, d_out, B, n_samples).total;
}

isopo_status isopo_sampled_coefficients(const void* X, const void* dY, isopo_dtype dtype, int64_t T, int d_in, int d_out,
                                        const int64_t* seq_offsets_host, int B, const int64_t* sample_rows_host,
                                        int n_samples, const float* A, float lambda, float* coeffs, float* F2, void* ws,
                                        size_t ws_bytes, int32_t* info, void* cuda_stream) {
  ApiRange nvtx_range("isopo_sampled_coefficients");
  if (!A || !coeffs || !info || !sample_rows_host) return ISOPO_ERR_INVALID_ARG;
  if (!(lambda >= 0.0f)) return ISOPO_ERR_INVALID_ARG;
  isopo_status s = check_layer_args(X, dY, dtype, T, d_in, d_out, seq_offsets_host, B, ISOPO_PATH_GRAM, ws);
  if (s != ISOPO_OK) return s;
  if (n_samples < 1 || n_samples > ISOPO_MAX_SAMPLES) return ISOPO_ERR_INVALID_ARG;
  for (int j = 0; j < n_samples; ++j)
    if (sample_rows_host[j] < 0 || sample_rows_host[j] >= T) return ISOPO_ERR_INVALID_ARG;
  const SampledLayout S = sampled_layout(dtype, T, d_in, d_out, B, n_samples, ws_bytes);
  if (ws_bytes < S.total) return ISOPO_ERR_WORKSPACE;
  const WsLayout L = ws_layout(dtype, T, d_in, d_out, B, ISOPO_PATH_GRAM);
  cudaStream_t st = (cudaStream_t)cuda_stream;
  char* w = (char*)ws;
  int32_t* tokseq = (int32_t*)(w + L.off_tokseq);
  const int64_t mt = (int64_t)n_samples * B * (dtype == ISOPO_F32 ? 2 : 1);  // M^T and its float64 denominator, in floats
  s = launch_prep(seq_offsets_host, B, T, (int64_t*)(w + L.off_offsets), tokseq,
                  Clear{{(float*)(w + S.off_mt), (float*)(w + S.off_den)}, {mt, 2}}, st);
  if (s != ISOPO_OK) return s;
  return sampled_coefficients(X, dY, dtype, T, d_in, d_out, tokseq, B, sample_rows_host, n_samples, w, S, A, lambda, coeffs,
                              F2, info, st);
}

isopo_status isopo_transform_advantages(const float* K, const float* A, int B, isopo_variant variant, float lambda,
                                        const float* opt_pqr_regs, float* coeffs, int32_t* info, void* cuda_stream) {
  ApiRange nvtx_range("isopo_transform_advantages");
  if (!K || !A || !coeffs || !info || B < 1) return ISOPO_ERR_INVALID_ARG;
  if ((int)variant < 0 || (int)variant > (int)ISOPO_VAR_NORMALISED_RAW) return ISOPO_ERR_INVALID_ARG;
  if (!(lambda >= 0.0f)) return ISOPO_ERR_INVALID_ARG;
  if (variant == ISOPO_VAR_GENERAL && !opt_pqr_regs) return ISOPO_ERR_INVALID_ARG;
  if (variant == ISOPO_VAR_INTERACTING && B > 256) return ISOPO_ERR_UNSUPPORTED;
  return transform(K, A, B, variant, lambda, opt_pqr_regs, nullptr, coeffs, info, (cudaStream_t)cuda_stream);
}

size_t isopo_transform_large_workspace_bytes(int B) {
  return B >= 1 && B <= ISOPO_MAX_LARGE_SEQS ? transform_large_workspace_bytes(B) : 0;
}

isopo_status isopo_transform_advantages_large(const float* K, const float* A, int B, float lambda, float* coeffs,
                                              void* workspace, size_t workspace_bytes, int32_t* info, void* cuda_stream) {
  ApiRange nvtx_range("isopo_transform_advantages_large");
  if (!K || !A || !coeffs || !info || !workspace || B < 1) return ISOPO_ERR_INVALID_ARG;
  if (!(lambda >= 0.0f) || ((uintptr_t)workspace & 15)) return ISOPO_ERR_INVALID_ARG;
  if (B > ISOPO_MAX_LARGE_SEQS) return ISOPO_ERR_UNSUPPORTED;
  if (workspace_bytes < transform_large_workspace_bytes(B)) return ISOPO_ERR_WORKSPACE;
  return transform_large(K, A, B, lambda, coeffs, (float*)workspace, info, (cudaStream_t)cuda_stream);
}

isopo_status isopo_reg_ema_update(const float* K, int B, float decay, float* state, void* cuda_stream) {
  ApiRange nvtx_range("isopo_reg_ema_update");
  if (!K || !state || B < 1 || !(decay >= 0.0f && decay < 1.0f)) return ISOPO_ERR_INVALID_ARG;
  return reg_ema_update(K, B, decay, state, (cudaStream_t)cuda_stream);
}

isopo_status isopo_transform_advantages_rel(const float* K, const float* A, int B, isopo_variant variant, float factor,
                                            const float* opt_pqr_factors, const float* state, float* coeffs,
                                            int32_t* info, void* cuda_stream) {
  ApiRange nvtx_range("isopo_transform_advantages_rel");
  if (!K || !A || !coeffs || !info || !state || B < 1) return ISOPO_ERR_INVALID_ARG;
  if ((int)variant < 0 || (int)variant > (int)ISOPO_VAR_NORMALISED_RAW) return ISOPO_ERR_INVALID_ARG;
  if (!(factor >= 0.0f)) return ISOPO_ERR_INVALID_ARG;
  if (variant == ISOPO_VAR_GENERAL && !opt_pqr_factors) return ISOPO_ERR_INVALID_ARG;
  if (variant == ISOPO_VAR_INTERACTING && B > 256) return ISOPO_ERR_UNSUPPORTED;
  return transform(K, A, B, variant, factor, opt_pqr_factors, state, coeffs, info, (cudaStream_t)cuda_stream);
}

isopo_status isopo_transform_advantages_batched(int n_layers, const float* const* K, const float* A, int B,
                                                isopo_variant variant, const float* lambda,
                                                const float* opt_pqr_regs, const float* const* states,
                                                float* const* coeffs, int32_t* info, void* cuda_stream) {
  ApiRange nvtx_range("isopo_transform_advantages_batched");
  if (n_layers < 1 || n_layers > ISOPO_MAX_BATCH) return ISOPO_ERR_INVALID_ARG;
  if (!K || !A || !lambda || !coeffs || !info || B < 1) return ISOPO_ERR_INVALID_ARG;
  if ((int)variant < 0 || (int)variant > (int)ISOPO_VAR_NORMALISED_RAW) return ISOPO_ERR_INVALID_ARG;
  if (variant == ISOPO_VAR_GENERAL && !opt_pqr_regs) return ISOPO_ERR_INVALID_ARG;
  if (variant == ISOPO_VAR_INTERACTING && B > 256) return ISOPO_ERR_UNSUPPORTED;
  for (int l = 0; l < n_layers; ++l) {
    if (!K[l] || !coeffs[l] || !(lambda[l] >= 0.0f) || (states && !states[l])) return ISOPO_ERR_INVALID_ARG;
  }
  return transform_batched(n_layers, K, A, B, variant, lambda, opt_pqr_regs, states, coeffs, info,
                           (cudaStream_t)cuda_stream);
}

isopo_status isopo_selftest_bounded_wait(int64_t limit_clocks, int32_t* info, int32_t* roles_at_teardown, void* cuda_stream) {
  ApiRange nvtx_range("isopo_selftest_bounded_wait");
  if (!info || !roles_at_teardown || limit_clocks < 1 || limit_clocks > ((int64_t)1 << 28)) return ISOPO_ERR_INVALID_ARG;
  return wait_probe((long long)limit_clocks, info, roles_at_teardown, (cudaStream_t)cuda_stream);
}

size_t isopo_spectral_workspace_bytes(void) { return spectral_workspace_bytes(); }

isopo_status isopo_transform_spectral(const float* K, const float* A, int B, float lambda, float rel_cutoff,
                                      float* coeffs, float* eigenvalues, void* ws, size_t ws_bytes, int32_t* info,
                                      void* cuda_stream) {
  ApiRange nvtx_range("isopo_transform_spectral");
  if (!K || !A || !coeffs || !ws || !info || B < 1) return ISOPO_ERR_INVALID_ARG;
  if (!(lambda >= 0.0f) || !(rel_cutoff >= 0.0f && rel_cutoff < 1.0f)) return ISOPO_ERR_INVALID_ARG;
  if ((uintptr_t)ws & 15) return ISOPO_ERR_INVALID_ARG;
  if (B > 256) return ISOPO_ERR_UNSUPPORTED;
  if (ws_bytes < spectral_workspace_bytes()) return ISOPO_ERR_WORKSPACE;
  return spectral(K, A, B, lambda, rel_cutoff, coeffs, eigenvalues, ws, info, (cudaStream_t)cuda_stream);
}

isopo_status isopo_transform_spectral_batched(int n_layers, const float* const* K, const float* A, int B,
                                              const float* lambda, float rel_cutoff, float* const* coeffs,
                                              float* const* eigenvalues, void* ws, size_t ws_bytes, int32_t* info,
                                              void* cuda_stream) {
  ApiRange nvtx_range("isopo_transform_spectral_batched");
  if (n_layers < 1 || n_layers > ISOPO_MAX_BATCH) return ISOPO_ERR_INVALID_ARG;
  if (!K || !A || !lambda || !coeffs || !ws || !info || B < 1) return ISOPO_ERR_INVALID_ARG;
  if (!(rel_cutoff >= 0.0f && rel_cutoff < 1.0f) || ((uintptr_t)ws & 15)) return ISOPO_ERR_INVALID_ARG;
  if (B > 256) return ISOPO_ERR_UNSUPPORTED;
  for (int l = 0; l < n_layers; ++l)
    if (!K[l] || !coeffs[l] || !(lambda[l] >= 0.0f)) return ISOPO_ERR_INVALID_ARG;
  if (ws_bytes < (size_t)n_layers * spectral_workspace_bytes()) return ISOPO_ERR_WORKSPACE;
  return spectral_batched(n_layers, K, A, B, lambda, rel_cutoff, coeffs, eigenvalues, ws, info,
                          (cudaStream_t)cuda_stream);
}

isopo_status isopo_weight_grad(const void* X, const void* dY, isopo_dtype dtype, int64_t T, int d_in, int d_out,
                               const float* coeffs, const int64_t* seq_offsets_host, int B, isopo_path path,
                               float* dW, float beta, void* ws, size_t ws_bytes, int32_t* info, void* cuda_stream) {
  ApiRange nvtx_range("isopo_weight_grad");
  if (!coeffs || !dW || !info) return ISOPO_ERR_INVALID_ARG;
  if (beta != 0.0f && beta != 1.0f) return ISOPO_ERR_INVALID_ARG;
  // the bf16 kernels write dW in pieces of 16 bytes and by TMA; refused here, before anything of dW is cleared
  if (dtype == ISOPO_BF16 && ((uintptr_t)dW & 15)) return ISOPO_ERR_INVALID_ARG;
  isopo_status s = check_layer_args(X, dY, dtype, T, d_in, d_out, seq_offsets_host, B, path, ws);
  if (s != ISOPO_OK) return s;
  const isopo_path rp = resolve_path(dtype, T, d_in, d_out, B, path);
  if (dtype == ISOPO_BF16 && rp == ISOPO_PATH_MATERIALISE && B > 256) return ISOPO_ERR_UNSUPPORTED;
  const WsLayout L = ws_layout(dtype, T, d_in, d_out, B, rp, ws_bytes);
  if (ws_bytes < L.total) return ISOPO_ERR_WORKSPACE;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  char* w = (char*)ws;
  if (rp == ISOPO_PATH_MATERIALISE) {
    // the kernels compare the tag isopo_layer_gram left with the one of this call and touch nothing on a mismatch
    const WsTag tag = make_ws_tag(dtype, T, d_in, d_out, B, seq_offsets_host);
    const WsTag* tag_dev = (const WsTag*)(w + L.off_tag);
    if (dtype == ISOPO_F32)
      return f32_combine((const float*)(w + L.off_G), (int64_t)d_in * d_out, L.n_pad, B, coeffs, dW, beta, tag_dev, tag, info, st);
    return bf16_combine(w + L.off_G, L, d_in, d_out, B, coeffs, dW, beta, tag_dev, tag, store_fmt(L, B, ws), info, st);
  }
  // GEMM over all tokens; the offsets travel again so that the call also works on its own
  const bool add = beta != 0.f;
  int64_t* off_dev = (int64_t*)(w + L.off_offsets);
  float* tokscale = (float*)(w + L.off_tokseq);  // one scale per token: a single independent load per row
  if (dtype == ISOPO_F32)
    return f32_weight_grad((const float*)X, (const float*)dY, T, d_in, d_out, seq_offsets_host, off_dev, coeffs, B, tokscale, dW, add, st);
  if (!bf16_weight_grad_uses_pairs(T, d_in, d_out, B))
    return bf16_weight_grad(X, dY, T, d_in, d_out, seq_offsets_host, off_dev, coeffs, B, tokscale, dW, add, info, st);
  if (bf16_weight_grad_fold_applies(T, d_in, d_out, B))
    return bf16_weight_grad_fold(X, dY, T, d_in, d_out, seq_offsets_host, off_dev, coeffs, B, dW, add, info, st);
  return bf16_weight_grad_pair(X, dY, T, d_in, d_out, seq_offsets_host, off_dev, coeffs, B, w + L.off_scaled, L.scaled_ld, dW, add, info, st);
}

}  // extern "C"
