// Token-sampled Fisher-norm estimator of Algorithm 1 (Sec. 2.2, "Efficient implementation"):
// with a0 = X[samples], g0 = dY[samples] (the rows the caller drew),
//   F_i^2 = sum_j (g0_j . G_i a0_j)^2 / sum_j (||g0_j|| ||a0_j||)^2 ,   c_i = A_i / sqrt(F_i^2 + lambda).
// G_i is never formed: g0_j . G_i a0_j = sum_{t in i} (g0_j . dY_t)(a0_j . x_t) =: M^T[j, i] (Eq. one), a
// rectangular cousin of the Gram route (tensor-core kernel in tc_gram.cu, float32 kernel in simt_f32.cu).
// This file holds what surrounds it: gathering the sampled rows (and the denominator, Eq. two)
// and the finishing step that turns M^T into F^2 and the coefficients.
#include <algorithm>

#include <cuda_bf16.h>

#include "isopo_internal.h"

namespace isopo {

namespace {

__device__ __forceinline__ float to_f32(float v) { return v; }
__device__ __forceinline__ float to_f32(__nv_bfloat16 v) { return __bfloat162float(v); }

__device__ __forceinline__ double block_sum_d(double v) {
  __shared__ double red[32];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) red[w] = v;
  __syncthreads();
  v = l < (blockDim.x >> 5) ? red[l] : 0.0;
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Copies one token row and returns this thread's share of its sum of squares.  Rows whose byte length and both
// addresses are multiples of 16 (every bfloat16 layer the library accepts) move as 16-byte vectors.
template <typename T>
__device__ __forceinline__ double copy_row_sq(const T* __restrict__ src, T* __restrict__ dst, int d) {
  constexpr int kVec = 16 / (int)sizeof(T);
  double acc = 0.0;
  if (d % kVec == 0 && (((uintptr_t)src | (uintptr_t)dst) & 15) == 0) {
    const uint4* s4 = reinterpret_cast<const uint4*>(src);
    uint4* d4 = reinterpret_cast<uint4*>(dst);
    for (int c = threadIdx.x; c < d / kVec; c += blockDim.x) {
      const uint4 v = __ldg(s4 + c);
      d4[c] = v;
      const T* e = reinterpret_cast<const T*>(&v);
      float part = 0.f;  // at most 8 squares of bfloat16 / 4 of float32 values: exact enough before the float64 sum
#pragma unroll
      for (int k = 0; k < kVec; ++k) {
        const float f = to_f32(e[k]);
        if (sizeof(T) == 2) part = fmaf(f, f, part); else acc += (double)f * (double)f;
      }
      if (sizeof(T) == 2) acc += (double)part;
    }
    return acc;
  }
  for (int c = threadIdx.x; c < d; c += blockDim.x) {
    const T v = src[c];
    dst[c] = v;
    const double f = (double)to_f32(v);
    acc += f * f;
  }
  return acc;
}

// The sample rows, as kernel arguments (token indices are below 2^31).
template <int kN> struct RowArgs { int32_t v[kN]; };

// Block j copies token row rows[j] of X and dY into a0[j], g0[j] and adds ||g0_j||^2 ||a0_j||^2 to *den.
template <typename T, int kN>
__global__ void __launch_bounds__(256) k_gather_samples(const T* __restrict__ X, const T* __restrict__ dY, int d_in,
                                                        int d_out, const __grid_constant__ RowArgs<kN> rows,
                                                        T* __restrict__ a0, int lda, T* __restrict__ g0, int ldg,
                                                        double* __restrict__ den) {
  pdl_wait();
  const int j = blockIdx.x;
  const int64_t t = rows.v[j];
  double na = copy_row_sq(X + t * d_in, a0 + (size_t)j * lda, d_in);
  double ng = copy_row_sq(dY + t * d_out, g0 + (size_t)j * ldg, d_out);
  na = block_sum_d(na);
  ng = block_sum_d(ng);
  if (threadIdx.x == 0) atomicAdd(den, na * ng);
}

// F_i^2 = sum_j M^T[j, i]^2 / den,  c_i = A_i / sqrt(F_i^2 + lambda).  A block of 32 x 8 threads serves 32
// sequences: thread (x, y) sums the samples j = y, y + 8, ... of sequence x (loads coalesced over x), the eight
// partial sums meet in shared memory.
constexpr int kFinishSlices = 8;
template <typename TM>
__global__ void __launch_bounds__(32 * kFinishSlices) k_sampled_finish(const TM* __restrict__ Mt, int n_samples, int B,
                                                                       const double* __restrict__ den,
                                                                       const float* __restrict__ A, float lambda,
                                                                       float* __restrict__ coeffs, float* __restrict__ F2) {
  pdl_wait();
  __shared__ double part[kFinishSlices][32];
  const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
  const int i = blockIdx.x * 32 + x;
  double s = 0.0;
  if (i < B)
    for (int j = y; j < n_samples; j += kFinishSlices) {
      const double m = (double)Mt[(size_t)j * B + i];
      s += m * m;
    }
  part[y][x] = s;
  __syncthreads();
  if (y != 0 || i >= B) return;
  s = 0.0;
#pragma unroll
  for (int k = 0; k < kFinishSlices; ++k) s += part[k][x];
  const double f2 = s / *den;
  if (F2) F2[i] = (float)f2;
  coeffs[i] = (float)((double)A[i] / sqrt(f2 + (double)lambda));
}

template <int kN, typename T>
isopo_status gather_with(const T* X, const T* dY, int d_in, int d_out, const int64_t* rows_host, int n_samples, T* a0, T* g0, const SampledLayout& S,
                         double* den, cudaStream_t st) {
  RowArgs<kN> rows;
  for (int j = 0; j < n_samples; ++j) rows.v[j] = (int32_t)rows_host[j];
  {
    LaunchScope scope(kIdSampledAux, st);
    launch(k_gather_samples<T, kN>, n_samples, 256, 0, st, X, dY, d_in, d_out, rows, a0, S.lda, g0, S.ldg, den);
  }
  ISOPO_CUDA_TRY(cudaGetLastError());
  return ISOPO_OK;
}
template <typename T>
isopo_status gather_samples(const T* X, const T* dY, int d_in, int d_out, const int64_t* rows_host, int n_samples, T* a0, T* g0,
                            const SampledLayout& S, double* den, cudaStream_t st) {
  return n_samples <= 256 ? gather_with<256>(X, dY, d_in, d_out, rows_host, n_samples, a0, g0, S, den, st)
                          : gather_with<ISOPO_MAX_SAMPLES>(X, dY, d_in, d_out, rows_host, n_samples, a0, g0, S, den, st);
}

}  // namespace

SampledLayout sampled_layout(isopo_dtype dtype, int64_t T, int d_in, int d_out, int B, int n_samples, size_t have) {
  const size_t elt = dtype == ISOPO_BF16 ? 2 : 4;
  const WsLayout L = ws_layout(dtype, T, d_in, d_out, B, ISOPO_PATH_GRAM, 0);  // offsets, token map (+ kacc), scaled operand
  auto lay = [&](bool lines) {
    SampledLayout S{};
    S.lda = lines ? line_pitch(d_in) : d_in;
    S.ldg = lines ? line_pitch(d_out) : d_out;
    // the scaled operand of the weight gradient behind it at lines as well; no copies of X and dY, which are read in place
    size_t p = lines ? L.off_scaled + align_up((size_t)2 * (size_t)T * (size_t)line_pitch(std::min(d_in, d_out)), 1024) : L.total;
    S.off_a0 = p;
    p = align_up(p + elt * (size_t)n_samples * S.lda, 1024);
    S.off_g0 = p;
    p = align_up(p + elt * (size_t)n_samples * S.ldg, 1024);
    S.off_mt = p;
    p = align_up(p + (dtype == ISOPO_BF16 ? sizeof(float) : sizeof(double)) * (size_t)n_samples * B, 1024);
    S.off_den = p;
    p = align_up(p + sizeof(double), 1024);
    S.total = p;
    return S;
  };
  // bf16: the tensor-core kernels' copies of the sample rows start at whole lines
  const SampledLayout S = lay(dtype == ISOPO_BF16);
  return have >= S.total ? S : lay(false);
}

isopo_status sampled_coefficients(const void* X, const void* dY, isopo_dtype dtype, int64_t T, int d_in, int d_out,
                                  const int32_t* tokseq, int B, const int64_t* rows_host, int n_samples, char* ws,
                                  const SampledLayout& S, const float* A, float lambda, float* coeffs, float* F2,
                                  int32_t* info, cudaStream_t st) {
  double* den = (double*)(ws + S.off_den);  // cleared, like M^T
  isopo_status s;
  if (dtype == ISOPO_F32) {
    float* a0 = (float*)(ws + S.off_a0);
    float* g0 = (float*)(ws + S.off_g0);
    double* Mt = (double*)(ws + S.off_mt);
    if ((s = gather_samples((const float*)X, (const float*)dY, d_in, d_out, rows_host, n_samples, a0, g0, S, den, st)) != ISOPO_OK) return s;
    s = f32_sampled((const float*)X, (const float*)dY, T, d_in, d_out, a0, g0, n_samples, tokseq, B, Mt, st);
    if (s != ISOPO_OK) return s;
    {
      LaunchScope scope(kIdSampledAux, st);
      launch(k_sampled_finish<double>, (B + 31) / 32, 32 * kFinishSlices, 0, st, Mt, n_samples, B, den, A, lambda, coeffs, F2);
    }
    ISOPO_CUDA_TRY(cudaGetLastError());
    return ISOPO_OK;
  }
  __nv_bfloat16* a0 = (__nv_bfloat16*)(ws + S.off_a0);
  __nv_bfloat16* g0 = (__nv_bfloat16*)(ws + S.off_g0);
  float* Mt = (float*)(ws + S.off_mt);
  s = gather_samples((const __nv_bfloat16*)X, (const __nv_bfloat16*)dY, d_in, d_out, rows_host, n_samples, a0, g0, S, den, st);
  if (s != ISOPO_OK) return s;
  s = bf16_sampled(X, dY, T, d_in, d_out, tokseq, B, a0, S.lda, g0, S.ldg, n_samples, Mt, info, st);
  if (s != ISOPO_OK) return s;
  {
    LaunchScope scope(kIdSampledAux, st);
    launch(k_sampled_finish<float>, (B + 31) / 32, 32 * kFinishSlices, 0, st, Mt, n_samples, B, den, A, lambda, coeffs, F2);
  }
  ISOPO_CUDA_TRY(cudaGetLastError());
  return ISOPO_OK;
}

}  // namespace isopo
