// Advantage transform: one CTA turns (K, A) into the per-sequence coefficients.
//   simple variants  - per-row sums of K in float64, a few rows per warp
//   interacting      - up to 128 sequences L D L^T in float64; more: blocked Cholesky of K + lambda*I with refinement
//                      (interacting_solve.cuh)
#include "cluster_solve.cuh"

namespace isopo {

namespace {

constexpr int kMaxB = 256;

// One launch serves up to ISOPO_MAX_BATCH layers that share A and the variant: CTA l works on layer l.
struct TransformBatch {
  TransformParams common;  // K, coeffs, lambda, rel_state are taken from the arrays below
  const float* K[ISOPO_MAX_BATCH];
  float* coeffs[ISOPO_MAX_BATCH];
  const float* rel_state[ISOPO_MAX_BATCH];
  float lambda[ISOPO_MAX_BATCH];
};

// The parameters of one layer of the batch, regularisers made absolute.
__device__ __forceinline__ TransformParams layer_params(const TransformBatch& batch, int layer) {
  TransformParams P = batch.common;
  P.K = batch.K[layer];
  P.coeffs = batch.coeffs[layer];
  P.rel_state = batch.rel_state[layer];
  P.lambda = batch.lambda[layer];
  if (P.rel_state) {
    // reg(val) = val + regularization * expectation(val) of the generalised re-scaling figure: each
    // regulariser is its factor times the running mean of the quantity it is added to
    const float eF = P.rel_state[0], eG = P.rel_state[1], eR = P.rel_state[2];
    switch (P.variant) {
      case ISOPO_VAR_NORMALISED:
      case ISOPO_VAR_NORMALISED_RAW: P.lambda *= eF; break;
      case ISOPO_VAR_DIRECTION: P.lambda *= eR; break;
      case ISOPO_VAR_EUCLID:
      case ISOPO_VAR_INTERACTING: P.lambda *= eG; break;  // mean eigenvalue of K = tr K / B = E[||G||^2]
      default: P.reg_F *= eF; P.reg_G *= eG; P.reg_rel *= eR;
    }
  }
  return P;
}

// Sums of squares of rows first .. last - 1 of K (four at a time, so that the loads of four rows are in flight), row by row to
// f(i, sum) in lane 0 of the calling warp.
template <bool kVec4, typename F>
__device__ __forceinline__ void row_square_sums(const float* __restrict__ K, int B, int first, int last, F f) {
  const int lane = threadIdx.x & 31;
  for (int i0 = first; i0 < last; i0 += 4) {
    double sq[4] = {};
    if (kVec4) {
#pragma unroll 2
      for (int j = lane * 4; j < B; j += 128) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const float4 v = __ldg(reinterpret_cast<const float4*>(K + (size_t)min(i0 + u, last - 1) * B + j));
          sq[u] += (double)v.x * v.x + (double)v.y * v.y + (double)v.z * v.z + (double)v.w * v.w;
        }
      }
    } else {
      for (int j = lane; j < B; j += 32)
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const double v = (double)__ldg(K + (size_t)min(i0 + u, last - 1) * B + j);
          sq[u] += v * v;
        }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) sq[u] = warp_sum(sq[u]);
    if (lane == 0)
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (i0 + u < last) f(i0 + u, sq[u]);
  }
}
// Sum over a block of kWarps warps, in the same order in every thread.
template <int kWarps>
__device__ __forceinline__ double block_total(double v, double* s_part) {
  v = warp_sum(v);
  if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = v;
  __syncthreads();
  double t = 0.0;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) t += s_part[w];
  return t;
}

// Simple variants.  Block (l, y): rows 32 y .. 32 y + 31 of layer l, four per warp; every block adds the trace up for
// itself.  Bound by latency: the seven layers of a block at 256 sequences took 25 us with one CTA per layer.
constexpr int kSimpleRows = 32;
__global__ void __launch_bounds__(256) k_transform_simple(const __grid_constant__ TransformBatch batch) {
  pdl_begin();
  const TransformParams P = layer_params(batch, blockIdx.x);
  __shared__ double s_part[8];
  const int B = P.B, tid = threadIdx.x, first = blockIdx.y * kSimpleRows;
  const float* __restrict__ K = P.K;
  if (P.variant == ISOPO_VAR_REINFORCE) {
    if (tid < kSimpleRows && first + tid < B) P.coeffs[first + tid] = P.A[first + tid];
    return;
  }
  double tr = 0.0;
  for (int i = tid; i < B; i += 256) tr += (double)__ldg(K + (size_t)i * B + i);
  __shared__ double s_sq[kSimpleRows];
  const int r0 = first + (tid >> 5) * 4;
  auto keep = [&](int i, double sq) { s_sq[i - first] = sq; };
  if (rows_in_float4(K, B)) row_square_sums<true>(K, B, r0, min(B, r0 + 4), keep);
  else row_square_sums<false>(K, B, r0, min(B, r0 + 4), keep);
  const double trace = block_total<8>(tr, s_part);
  const int i = first + tid;
  if (tid >= kSimpleRows || i >= B) return;
  const double sq = s_sq[tid], n2 = (double)K[(size_t)i * B + i];
  const double F2 = P.variant == ISOPO_VAR_NORMALISED_RAW ? sq / (double)B : sq / trace;
  const double a = (double)P.A[i], lam = (double)P.lambda;
  double c;
  switch (P.variant) {
    case ISOPO_VAR_NORMALISED:
    case ISOPO_VAR_NORMALISED_RAW: c = a / sqrt(F2 + lam); break;
    case ISOPO_VAR_DIRECTION: c = a / (F2 / n2 + lam); break;
    case ISOPO_VAR_EUCLID: c = a / sqrt(n2 + lam); break;
    default: {  // ISOPO_VAR_GENERAL
      const double eps = 1e-8;
      const double rF = sqrt(F2 + (double)P.reg_F + eps);
      const double rG = sqrt(n2 + (double)P.reg_G + eps);
      const double rR = sqrt(F2 / n2 + (double)P.reg_rel + eps);
      c = a * pow(rF, (double)P.p) * pow(rG, (double)P.q) * pow(rR, (double)P.r);
    }
  }
  P.coeffs[i] = (float)c;
}

// Interacting variant, up to 128 sequences: (K + lambda I) c = A in float64 by block elimination with 2 x 2 pivots (a
// block L D L^T), one CTA per layer.  Thread (ty, tx) of a 16 x 16 grid keeps the elements (ty + 16 p, tx + 16 q) in
// registers.  A step publishes two columns C in shared memory, and after ONE barrier everybody forms the rows of
// T = C P^-1, P the pivot, that it needs and subtracts T C^T from its elements; the right-hand side rides along, one
// element per thread.  T stays in shared memory for the backward solve, one warp's work.  An odd last row gets a unit row.
// Bound by latency: a step's barrier, shared load, reciprocal and some ten dependent float64 operations.  Single columns
// (one reciprocal and one barrier each) took 16.4 us at 64 and 41 us at 128 sequences, this 14.7 and 36.9.  In float64 the
// solution needs no refinement; the blocked float32 kernel below, which does, takes 21.5 and 39 us when its unrolled code
// is in the instruction cache and about twice that when a GEMM ran before it.
// 1 / d by Newton's iteration from the hardware's approximation (about 20 bits; twice gives all 53).
__device__ __forceinline__ double newton_rcp(double d) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(d));
  r = fma(r, fma(-d, r, 1.0), r);
  return fma(r, fma(-d, r, 1.0), r);
}
template <int kA>
__global__ void __launch_bounds__(256) k_transform_small(const __grid_constant__ TransformBatch batch) {
  pdl_begin();
  extern __shared__ __align__(16) double smem_d[];
  const TransformParams P = layer_params(batch, blockIdx.x);
  const int B = P.B, n = B + (B & 1), tid = threadIdx.x, ty = tid >> 4, tx = tid & 15, pitch = n + 1;
  double* T = smem_d;                            // [k * pitch + i]: T(i, k), i > k
  double* y = T + (size_t)n * pitch;             // D^-1 y
  double2* col = reinterpret_cast<double2*>(y + n);  // [2][n]: the two columns of a step, two buffers
  double2* ycol = col + 2 * n;                   // [2]: the right-hand side's two elements
  double a[kA][kA];
#pragma unroll
  for (int p = 0; p < kA; ++p)
#pragma unroll
    for (int q = 0; q <= p; ++q) {
      const int i = ty + 16 * p, j = tx + 16 * q;
      a[p][q] = i < B && j < B ? (double)__ldg(P.K + (size_t)i * B + j) + (i == j ? (double)P.lambda : 0.0) : i == j ? 1.0 : 0.0;
    }
  int iy[kA], jx[kA];  // this thread's rows and columns, kept inside the matrix
#pragma unroll
  for (int p = 0; p < kA; ++p) { iy[p] = min(ty + 16 * p, n - 1); jx[p] = min(tx + 16 * p, n - 1); }
  double rhs = tid < B ? (double)P.A[tid] : 0.0;
  int fail = 0;
#pragma unroll
  for (int q = 0; q < kA; ++q) {
#pragma unroll 1
    for (int k = 16 * q; k < min(n, 16 * q + 16); k += 2) {
      double2* c = col + ((k >> 1) & 1) * n;
      double2* yc = ycol + ((k >> 1) & 1);
      if ((tx & ~1) == (k & 15)) {
        double* half = reinterpret_cast<double*>(c) + (tx & 1);
#pragma unroll
        for (int p = q; p < kA; ++p) {
          const int i = ty + 16 * p;
          if (i >= k && i < n) half[2 * i] = a[p][q];
        }
      }
      if ((tid & ~1) == k) reinterpret_cast<double*>(yc)[tid & 1] = rhs;
      __syncthreads();
      const double2 r0 = c[k], r1 = c[k + 1];  // P = [r0.x r1.x; r1.x r1.y]
      const double det = fma(r0.x, r1.y, -(r1.x * r1.x));
      if (!(r0.x > 0.0)) fail = k + 1;
      else if (!(det > 0.0)) fail = k + 2;
      if (fail) break;  // the same in every thread
      const double inv = newton_rcp(det);
      const double p00 = r1.y * inv, p01 = -r1.x * inv, p11 = r0.x * inv;  // P^-1
      const double2 yk = *yc;
      if (tid == 0) { y[k] = p00 * yk.x + p01 * yk.y; y[k + 1] = p01 * yk.x + p11 * yk.y; }
      double2 cj[kA];  // rows and columns up to k + 1 take part with whatever they hold: nothing reads them again
#pragma unroll
      for (int p = q; p < kA; ++p) cj[p] = c[jx[p]];
#pragma unroll
      for (int p = q; p < kA; ++p) {
        const double2 ci = c[iy[p]];
        const double t0 = fma(p00, ci.x, p01 * ci.y), t1 = fma(p01, ci.x, p11 * ci.y);
#pragma unroll
        for (int r = q; r <= p; ++r) a[p][r] = fma(-t1, cj[r].y, fma(-t0, cj[r].x, a[p][r]));
        if (tx < 2 && ty + 16 * p < n) T[(size_t)(k + tx) * pitch + ty + 16 * p] = tx ? t1 : t0;
      }
      if (tid > k + 1 && tid < B) {
        const double2 ci = c[tid];
        rhs = fma(-fma(p01, ci.x, p11 * ci.y), yk.y, fma(-fma(p00, ci.x, p01 * ci.y), yk.x, rhs));
      }
    }
    if (fail) break;
  }
  if (fail) {
    if (tid == 0) atomicCAS(P.info, 0, fail + ((int)blockIdx.x << 16));
    if (tid < B) P.coeffs[tid] = 0.f;
    return;
  }
  __syncthreads();
  if (tid >= 32) return;
  // x_J = P_J^-1 y_J - sum over later rows k of T(k, J) x_k; lane l holds the elements l + 32 c
  constexpr int kC = (kA + 1) / 2;
  double x[kC], l0[kC], l1[kC];
#pragma unroll
  for (int c = 0; c < kC; ++c) {
    const int j = tid + 32 * c;
    x[c] = j < n ? y[j] : 0.0;
    l0[c] = j < n - 2 ? T[(size_t)j * pitch + n - 2] : 0.0;
    l1[c] = j < n - 2 ? T[(size_t)j * pitch + n - 1] : 0.0;
  }
#pragma unroll
  for (int c = kC - 1; c >= 0; --c) {
#pragma unroll 1
    for (int k = min(n, 32 * c + 32) - 2; k >= 32 * c; k -= 2) {
      const double x0 = __shfl_sync(0xffffffffu, x[c], k & 31), x1 = __shfl_sync(0xffffffffu, x[c], (k & 31) + 1);
#pragma unroll
      for (int b = 0; b <= c; ++b) {
        const int j = tid + 32 * b;
        x[b] = fma(-l1[b], x1, fma(-l0[b], x0, x[b]));
        l0[b] = j < k - 2 ? T[(size_t)j * pitch + k - 2] : 0.0;
        l1[b] = j < k - 2 ? T[(size_t)j * pitch + k - 1] : 0.0;
      }
    }
  }
#pragma unroll
  for (int c = 0; c < kC; ++c)
    if (tid + 32 * c < B) P.coeffs[tid + 32 * c] = (float)x[c];
}
constexpr int kMaxSmallB = 128;
inline size_t small_smem_bytes(int B) {
  const size_t n = (size_t)B + (B & 1);
  return sizeof(double) * (n * (n + 1) + n + 4 * n + 4);
}

// Interacting variant, 129 to 256 sequences: one CTA per layer, the factor in shared memory.
__global__ void __launch_bounds__(kSolveThreads, 1) k_transform(const __grid_constant__ TransformBatch batch) {
  pdl_begin();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const TransformParams P = layer_params(batch, blockIdx.x);
  __shared__ double s_trace, s_res;
  __shared__ int s_fail;
  const SolveSmem m = solve_smem(smem_raw, P.B);
  interacting_solve(P, m.Lb, m.InvD, m.vec, m.sol, m.rdiag, s_trace, s_res, s_fail, (int)blockIdx.x);
}

// 257 to 1024 sequences: a cluster of sixteen, the factor's blocks also in a workspace that stays in the L2 (2.1 MB at 1024).
// Where no such cluster can be placed (a context that has a part of the SMs): transform_one_cta.cu.
constexpr int kMaxLargeB = ISOPO_MAX_LARGE_SEQS;
constexpr int kLargeCluster = 16;
__global__ void __launch_bounds__(kClThreads, 1) k_transform_large(const TransformParams P, float* scratch) {
  pdl_begin();
  extern __shared__ __align__(128) unsigned char smem_raw[];
  cluster_solve<kLargeCluster>(P, scratch, smem_raw, 0);
}

// Running means for the relative regulariser.  state = {E[F^2], E[||G||^2], E[F^2 / ||G||^2], number of updates};
// the first update stores this microbatch's means, later ones blend: s <- decay * s + (1 - decay) * mean.
// One pass: F_i^2 = sum_j K_ij^2 / tr K, so all three means follow from sums of row sums.
// The grid is one cluster, which shares the rows (four to a warp at a time), and its first CTA adds up.  Bound by latency: 156 sequences 7.4 -> 4.9 us against
// one CTA of 1024 threads, 255 9.1 -> 6.4, 1024 49.8 -> 20.2; up to 100 sequences 4.9 either way (the call's host time).
constexpr int kEmaThreads = 256;
constexpr int kEmaCluster = 8;
__global__ void __launch_bounds__(kEmaThreads)
k_reg_ema(const float* __restrict__ K, int B, float decay, float* __restrict__ state) {
  pdl_begin();
  constexpr int kWarps = kEmaThreads / 32;
  __shared__ double s_part[kEmaCluster * kWarps][3];  // first CTA: of every warp of the cluster
  const int tid = threadIdx.x, lane = tid & 31, rank = (int)tc::cluster_ctarank(), warp = rank * kWarps + (tid >> 5);
  const int ctas = gridDim.x, step = ctas * kWarps * 4;
  double tr = 0.0, f2 = 0.0, rel = 0.0;
  for (int i = rank * kEmaThreads + tid; i < B; i += ctas * kEmaThreads) tr += (double)__ldg(K + (size_t)i * B + i);
  auto add = [&](int i, double sq) {
    f2 += sq;
    rel += sq / (double)__ldg(K + (size_t)i * B + i);
  };
  if (rows_in_float4(K, B))  // outside the row loop: inside it 1024 sequences took 72 us instead of 53 in one CTA
    for (int i0 = warp * 4; i0 < B; i0 += step) row_square_sums<true>(K, B, i0, min(B, i0 + 4), add);
  else
    for (int i0 = warp * 4; i0 < B; i0 += step) row_square_sums<false>(K, B, i0, min(B, i0 + 4), add);
  tr = warp_sum(tr);
  cl_arrive();
  cl_wait();  // the first CTA runs
  if (lane == 0) {
    const double part[3] = {tr, f2, rel};
#pragma unroll
    for (int k = 0; k < 3; ++k) st_cluster_f64(tc::map_to_cta(tc::smem_u32(&s_part[warp][k]), 0), part[k]);
  }
  __syncwarp();  // the barrier wants the warp together
  cl_arrive();
  cl_wait();
  if (rank != 0 || tid >= 32) return;
  double sum[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) sum[k] = warp_sum((lane < ctas * kWarps ? s_part[lane][k] : 0.0) + (lane + 32 < ctas * kWarps ? s_part[lane + 32][k] : 0.0));
  static_assert(kEmaCluster * kWarps == 64, "two partial sums to a lane");
  const double trace = sum[0];
  if (lane == 0) {
    const double m[3] = {sum[1] / trace / B, trace / B, sum[2] / trace / B};
    const bool first = state[3] == 0.f;
    for (int k = 0; k < 3; ++k)
      state[k] = (float)(first ? m[k] : (double)decay * (double)state[k] + (1.0 - (double)decay) * m[k]);
    state[3] += 1.f;
  }
}

}  // namespace

isopo_status reg_ema_update(const float* K, int B, float decay, float* state, cudaStream_t st) {
  const unsigned ctas = B <= 4 * kEmaThreads / 32 ? 1 : (unsigned)placed_cluster(kEmaCluster);  // one has a row for every warp
  {
    LaunchScope scope(kIdTransform, st);
    launch_cluster(k_reg_ema, ctas, ctas, kEmaThreads, 0, st, K, B, decay, state);
  }
  ISOPO_CUDA_TRY(cudaGetLastError());
  return ISOPO_OK;
}

isopo_status transform_batched(int n, const float* const* K, const float* A, int B, isopo_variant v, const float* lambda,
                               const float* g, const float* const* rel_state, float* const* coeffs, int32_t* info,
                               cudaStream_t st) {
  TransformBatch T{};
  TransformParams& P = T.common;
  P.A = A; P.info = info; P.B = B; P.variant = (int)v;
  if (v == ISOPO_VAR_GENERAL) { P.p = g[0]; P.q = g[1]; P.r = g[2]; P.reg_F = g[3]; P.reg_G = g[4]; P.reg_rel = g[5]; }
  for (int l = 0; l < n; ++l) {
    T.K[l] = K[l];
    T.coeffs[l] = coeffs[l];
    T.rel_state[l] = rel_state ? rel_state[l] : nullptr;
    T.lambda[l] = lambda[l];
  }
  if (v != ISOPO_VAR_INTERACTING) {
    LaunchScope scope(kIdTransform, st);
    launch(k_transform_simple, dim3(n, (B + kSimpleRows - 1) / kSimpleRows), 256, 0, st, T);
  } else if (B <= kMaxSmallB) {
    auto kernel = B <= 16 ? k_transform_small<1> : B <= 32 ? k_transform_small<2> : B <= 64 ? k_transform_small<4> : k_transform_small<8>;
    const size_t smem = small_smem_bytes(B);
    if (smem > 48 * 1024) ISOPO_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
    LaunchScope scope(kIdTransform, st);
    launch(kernel, n, 256, smem, st, T);
  } else {
    if (B > kMaxB) return ISOPO_ERR_UNSUPPORTED;
    ISOPO_CUDA_TRY(cudaFuncSetAttribute(k_transform, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
    LaunchScope scope(kIdTransform, st);
    launch(k_transform, n, kSolveThreads, solve_smem_bytes(B), st, T);
  }
  ISOPO_CUDA_TRY(cudaGetLastError());
  return ISOPO_OK;
}

size_t transform_large_workspace_bytes(int B) {
  const size_t nb = (size_t)(B + kNB - 1) / kNB;
  return sizeof(float) * (nb * (nb + 1) / 2) * kBlk;
}

isopo_status transform_large(const float* K, const float* A, int B, float lambda, float* coeffs, float* scratch,
                             int32_t* info, cudaStream_t st) {
  if (B < 1 || B > kMaxLargeB) return ISOPO_ERR_UNSUPPORTED;
  if (B <= kMaxB) return transform(K, A, B, ISOPO_VAR_INTERACTING, lambda, nullptr, nullptr, coeffs, info, st);
  TransformParams P{};
  P.K = K; P.A = A; P.coeffs = coeffs; P.info = info; P.B = B; P.variant = (int)ISOPO_VAR_INTERACTING; P.lambda = lambda;
  ISOPO_CUDA_TRY(cudaFuncSetAttribute(k_transform_large, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
  ISOPO_CUDA_TRY(cudaFuncSetAttribute(k_transform_large, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kLargeCluster);
  cfg.blockDim = dim3(kClThreads);
  cfg.dynamicSmemBytes = cl_smem_bytes<kLargeCluster>(B);
  cfg.stream = st;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = kLargeCluster; attr.val.clusterDim.y = 1; attr.val.clusterDim.z = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  int clusters = 0;  // asked at every call: a device's contexts may have different SMs
  ISOPO_CUDA_TRY(cudaOccupancyMaxActiveClusters(&clusters, k_transform_large, &cfg));
  if (clusters == 0) return transform_one_cta(K, A, B, lambda, coeffs, scratch, info, st);
  {
    LaunchScope scope(kIdTransform, st);
    ISOPO_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_transform_large, P, scratch));
  }
  ISOPO_CUDA_TRY(cudaGetLastError());
  return ISOPO_OK;
}

isopo_status transform(const float* K, const float* A, int B, isopo_variant v, float lambda, const float* g,
                       const float* rel_state, float* coeffs, int32_t* info, cudaStream_t st) {
  return transform_batched(1, &K, A, B, v, &lambda, g, rel_state ? &rel_state : nullptr, &coeffs, info, st);
}

}  // namespace isopo
