// Advantage transform: one CTA turns (K, A) into the per-sequence coefficients.
//   simple variants  - per-row sums of K in float64, one warp per row
//   interacting      - blocked Cholesky of K + lambda*I with refinement (interacting_solve.cuh)
#include "interacting_solve.cuh"

namespace isopo {

namespace {

constexpr int kThreads = kSolveThreads;
constexpr int kMaxB = 256;

// One launch serves up to ISOPO_MAX_BATCH layers that share A and the variant: CTA l works on layer l.
struct TransformBatch {
  TransformParams common;  // K, coeffs, lambda, rel_state are taken from the arrays below
  const float* K[ISOPO_MAX_BATCH];
  float* coeffs[ISOPO_MAX_BATCH];
  const float* rel_state[ISOPO_MAX_BATCH];
  float lambda[ISOPO_MAX_BATCH];
};

__global__ void __launch_bounds__(kThreads) k_transform(const __grid_constant__ TransformBatch batch) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  TransformParams P = batch.common;
  P.K = batch.K[blockIdx.x];
  P.coeffs = batch.coeffs[blockIdx.x];
  P.rel_state = batch.rel_state[blockIdx.x];
  P.lambda = batch.lambda[blockIdx.x];
  __shared__ double s_trace, s_res;
  __shared__ int s_fail;
  const int B = P.B, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = kThreads / 32;
  const float* __restrict__ K = P.K;
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

  if (P.variant == ISOPO_VAR_REINFORCE) {
    for (int i = tid; i < B; i += kThreads) P.coeffs[i] = P.A[i];
    return;
  }

  if (P.variant != ISOPO_VAR_INTERACTING) {
    // trace of K
    double tr = 0.0;
    for (int i = tid; i < B; i += kThreads) tr += (double)K[(size_t)i * B + i];
    tr = warp_sum(tr);
    if (tid == 0) s_trace = 0.0;
    __syncthreads();
    if (lane == 0) atomicAdd(&s_trace, tr);
    __syncthreads();
    const double trace = s_trace;
    for (int i = warp; i < B; i += nwarps) {
      double sq = 0.0;
      for (int j = lane; j < B; j += 32) {
        const double kij = (double)K[(size_t)i * B + j];
        sq += kij * kij;
      }
      sq = warp_sum(sq);
      if (lane == 0) {
        const double n2 = (double)K[(size_t)i * B + i];
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
    }
    return;
  }

  // ---------------- interacting: (K + lambda I) c = A ----------------
  const SolveSmem m = solve_smem(smem_raw, B);
  interacting_solve<false>(P, m.Lb, m.InvD, m.vec, m.sol, m.rdiag, s_trace, s_res, s_fail, (int)blockIdx.x);
}

// The interacting variant for more sequences than the shared-memory kernel holds: the block triangle (2.1 MB at
// 1024 sequences) lives in a workspace that stays in the L2, everything else as above.  One CTA.
constexpr int kMaxLargeB = ISOPO_MAX_LARGE_SEQS;
__global__ void __launch_bounds__(kThreads) k_transform_large(const TransformParams P, float* scratch) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double s_trace, s_res;
  __shared__ int s_fail;
  const int nb = (P.B + kNB - 1) / kNB, Bp = nb * kNB;
  float* InvD = reinterpret_cast<float*>(smem_raw);         // nb inverse diagonal factors
  float* vec = InvD + (size_t)nb * kBlk;                    // Bp floats
  double* sol = reinterpret_cast<double*>(vec + Bp);        // Bp doubles
  float* rdiag = reinterpret_cast<float*>(sol + Bp);        // Bp floats
  interacting_solve<true>(P, scratch, InvD, vec, sol, rdiag, s_trace, s_res, s_fail, 0);
}

// Running means for the relative regulariser.  state = {E[F^2], E[||G||^2], E[F^2 / ||G||^2], number of updates};
// the first update stores this microbatch's means, later ones blend: s <- decay * s + (1 - decay) * mean.
__global__ void __launch_bounds__(kThreads) k_reg_ema(const float* __restrict__ K, int B, float decay,
                                                      float* __restrict__ state) {
  __shared__ double s_trace, s_f2, s_rel;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = kThreads / 32;
  double tr = 0.0;
  for (int i = tid; i < B; i += kThreads) tr += (double)K[(size_t)i * B + i];
  tr = warp_sum(tr);
  if (tid == 0) { s_trace = 0.0; s_f2 = 0.0; s_rel = 0.0; }
  __syncthreads();
  if (lane == 0) atomicAdd(&s_trace, tr);
  __syncthreads();
  const double trace = s_trace;
  double f2_sum = 0.0, rel_sum = 0.0;
  for (int i = warp; i < B; i += nwarps) {
    double sq = 0.0;
    for (int j = lane; j < B; j += 32) {
      const double kij = (double)K[(size_t)i * B + j];
      sq += kij * kij;
    }
    sq = warp_sum(sq);
    const double F2 = sq / trace;
    f2_sum += F2;
    rel_sum += F2 / (double)K[(size_t)i * B + i];
  }
  if (lane == 0) { atomicAdd(&s_f2, f2_sum); atomicAdd(&s_rel, rel_sum); }
  __syncthreads();
  if (tid == 0) {
    const double m[3] = {s_f2 / B, trace / B, s_rel / B};
    const bool first = state[3] == 0.f;
    for (int k = 0; k < 3; ++k)
      state[k] = (float)(first ? m[k] : (double)decay * (double)state[k] + (1.0 - (double)decay) * m[k]);
    state[3] += 1.f;
  }
}

}  // namespace

isopo_status reg_ema_update(const float* K, int B, float decay, float* state, cudaStream_t st) {
  {
    LaunchScope scope(kIdTransform, st);
    k_reg_ema<<<1, kThreads, 0, st>>>(K, B, decay, state);
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
  size_t smem = 0;
  if (v == ISOPO_VAR_INTERACTING) {
    if (B > kMaxB) return ISOPO_ERR_UNSUPPORTED;
    smem = solve_smem_bytes(B);
    ISOPO_CUDA_TRY(cudaFuncSetAttribute(k_transform, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
  }
  {
    LaunchScope scope(kIdTransform, st);
    k_transform<<<n, kThreads, smem, st>>>(T);
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
  TransformParams P{};
  P.K = K; P.A = A; P.coeffs = coeffs; P.info = info; P.B = B; P.variant = (int)ISOPO_VAR_INTERACTING; P.lambda = lambda;
  const size_t nb = (size_t)(B + kNB - 1) / kNB;
  const size_t smem = sizeof(float) * (nb * kBlk + 2 * nb * kNB) + sizeof(double) * nb * kNB;
  ISOPO_CUDA_TRY(cudaFuncSetAttribute(k_transform_large, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
  {
    LaunchScope scope(kIdTransform, st);
    k_transform_large<<<1, kThreads, smem, st>>>(P, scratch);
  }
  ISOPO_CUDA_TRY(cudaGetLastError());
  return ISOPO_OK;
}

isopo_status transform(const float* K, const float* A, int B, isopo_variant v, float lambda, const float* g,
                       const float* rel_state, float* coeffs, int32_t* info, cudaStream_t st) {
  return transform_batched(1, &K, A, B, v, &lambda, g, rel_state ? &rel_state : nullptr, &coeffs, info, st);
}

}  // namespace isopo
