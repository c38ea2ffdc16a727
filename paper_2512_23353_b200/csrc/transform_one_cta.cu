// Interacting solve for 257 to 1024 sequences by one CTA, the factor in a workspace that stays in the L2: what
// isopo_transform_advantages_large does where a cluster of sixteen CTAs (transform.cu) cannot be placed, i.e. in a context that
// has a part of the SMs.  512 sequences 398 us (the cluster 148), 1024 2182 us (338).  A file of its own: in transform.cu the
// cluster's kernel, whose helpers it shares, took 4 us longer at 1024 sequences.
#include "interacting_solve.cuh"

namespace isopo {

namespace {

__global__ void __launch_bounds__(kSolveThreads) k_transform_one_cta(const TransformParams P, float* scratch) {
  pdl_begin();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double s_trace, s_res;
  __shared__ int s_fail;
  const int nb = (P.B + kNB - 1) / kNB, Bp = nb * kNB;
  float* InvD = reinterpret_cast<float*>(smem_raw);   // nb inverse diagonal factors
  float* vec = InvD + (size_t)nb * kBlk;              // Bp floats
  double* sol = reinterpret_cast<double*>(vec + Bp);  // Bp doubles
  float* rdiag = reinterpret_cast<float*>(sol + Bp);  // Bp floats
  interacting_solve<kSolveThreads, false>(P, scratch, InvD, vec, sol, rdiag, s_trace, s_res, s_fail, 0);
}

}  // namespace

isopo_status transform_one_cta(const float* K, const float* A, int B, float lambda, float* coeffs, float* scratch, int32_t* info,
                               cudaStream_t st) {
  TransformParams P{};
  P.K = K; P.A = A; P.coeffs = coeffs; P.info = info; P.B = B; P.variant = (int)ISOPO_VAR_INTERACTING; P.lambda = lambda;
  const size_t nb = (size_t)(B + kNB - 1) / kNB;
  const size_t smem = sizeof(float) * (nb * kBlk + 2 * nb * kNB) + sizeof(double) * nb * kNB;
  ISOPO_CUDA_TRY(cudaFuncSetAttribute(k_transform_one_cta, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
  {
    LaunchScope scope(kIdTransform, st);
    launch(k_transform_one_cta, 1, kSolveThreads, smem, st, P, scratch);
  }
  ISOPO_CUDA_TRY(cudaGetLastError());
  return ISOPO_OK;
}

}  // namespace isopo
