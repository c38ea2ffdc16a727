// Interacting solve (K + lambda I) c = A by one CTA: blocked Cholesky (float32, 32 x 32 blocks, warp-level diagonal
// factorisation), blocked triangular solves, then up to two refinement rounds with float64 residuals taken from the
// float32 K, stopped once the relative residual is below 1e-7.  Used by the advantage transform (transform.cu) and by
// the spectral variant (spectral.cu).
#pragma once

#include "isopo_internal.h"

namespace isopo {

namespace {

constexpr int kSolveThreads = 512;

struct TransformParams {
  const float* K;
  const float* A;
  float* coeffs;
  int32_t* info;
  int B;
  int variant;
  float lambda;
  float p, q, r, reg_F, reg_G, reg_rel;
  const float* rel_state;  // NULL, or the running means {E[F^2], E[||G||^2], E[F^2/||G||^2], updates}: the
                           // regularisers above are then factors of these (relative regularisation)
};

// Whether the rows of a B x B matrix can be read 16 bytes at a time: callers may keep several K in one buffer, so its address
// is a multiple of 4 bytes and no more.
__device__ __forceinline__ bool rows_in_float4(const float* K, int B) {
  return (B & 3) == 0 && (reinterpret_cast<uintptr_t>(K) & 15) == 0;
}

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// ---------------------------------------------------------------------------------------------
// Interacting variant: blocked Cholesky in shared memory.
//
// K + lambda*I is held as 32 x 32 blocks (lower block triangle, block (I,J) at slot I(I+1)/2+J),
// every block column-major: element (r, c) at [c*32 + r], so that a warp whose lane owns row r
// reads a block column without bank conflicts and 4 consecutive rows form one float4.
// Per block column J:  (1) one warp per block below the diagonal solves X L_JJ^T = A_IJ by
// substitution (lane = row), while a spare warp inverts L_JJ for the solve phase;  (2) one warp per
// trailing block does the rank-32 update with 4 x 8 register tiles; block (J+1, J+1) is updated
// first, by all warps together, and warp 0 then factors it in registers (shuffles), so the serial
// pivot chain of the next column runs beside the other warps' updates instead of after them.  The triangular solves with the
// right-hand side use the stored inverses of the diagonal blocks.
// ---------------------------------------------------------------------------------------------
constexpr int kNB = 32;
constexpr int kBlk = kNB * kNB;

__device__ __forceinline__ int blk_slot(int I, int J) { return I * (I + 1) / 2 + J; }

// Column sums over the warp: on entry lane l holds r[c] = M[l][c]; on return r[0] of lane c holds
// sum_l M[l][c].  Recursive halving: 31 shuffles for all 32 sums.
__device__ __forceinline__ float warp_column_sums(float (&r)[kNB]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int idx = 0; idx < o; ++idx) {
      const float send = up ? r[idx] : r[idx + o];
      const float keep = up ? r[idx + o] : r[idx];
      r[idx] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  return r[0];
}

// Pointer types of the block helpers.  kShared: every block lies in this CTA's shared memory, is written by one warp at a time, and a
// lane of a helper reads of it what others left before the call or what it wrote itself, so the pointers may be restrict-qualified
// (4 % of the solve at 256 sequences).  Otherwise a block may be global memory that another warp or SM wrote earlier in the same
// kernel: plain loads only, never the read-only path.
template <bool kShared> struct BlkPtr { typedef float* __restrict__ rw; typedef const float* __restrict__ ro; };
template <> struct BlkPtr<false> { typedef float* rw; typedef const float* ro; };

// Factors the 32 x 32 diagonal block D (column-major, symmetric input) in place into its lower
// Cholesky factor and writes 1 / L_kk to rd[k].  One warp.  D is not restrict-qualified: in shared memory its lanes read columns that the
// others have just written, and a load through such a pointer could be moved ahead of the __syncwarp between.
// Returns 0, or the 1-based local index of the first non-positive pivot.
template <bool kShared = true>
__device__ __noinline__ int warp_factor_diag(float* D, float* __restrict__ rd) {
  const int lane = threadIdx.x & 31;
  float r[kNB];
#pragma unroll
  for (int c = 0; c < kNB; ++c) r[c] = D[c * kNB + lane];  // row `lane`
  int fail = 0;
  float rdiag = 0.f;  // 1 / L[lane][lane]
  float d = __shfl_sync(0xffffffffu, r[0], 0), rs = rsqrtf(d);
#pragma unroll
  for (int k = 0; k < kNB; ++k) {
    if (!(d > 0.f) && fail == 0) fail = k + 1;
    if (lane == k) rdiag = rs;
    r[k] = lane == k ? d * rs : r[k] * rs;  // L[lane][k] (rows above k hold junk, never used)
    if (kShared) {
      D[k * kNB + lane] = k <= lane ? r[k] : 0.f;
      __syncwarp();
    }
    // the next pivot first: its chain (two shuffles, a reciprocal root) runs under the updates of the columns behind it, which read
    // column k from shared memory four entries at a time
    if (k + 1 < kNB) {
      r[k + 1] = fmaf(-r[k], __shfl_sync(0xffffffffu, r[k], k + 1), r[k + 1]);
      d = __shfl_sync(0xffffffffu, r[k + 1], k + 1);
      rs = rsqrtf(d);
    }
    if (kShared) {
#pragma unroll
      for (int j = (k + 2) & ~3; j < kNB; j += 4) {
        const float4 l = *reinterpret_cast<const float4*>(D + k * kNB + j);
        if (j > k + 1) r[j] = fmaf(-r[k], l.x, r[j]);
        if (j + 1 > k + 1) r[j + 1] = fmaf(-r[k], l.y, r[j + 1]);
        if (j + 2 > k + 1) r[j + 2] = fmaf(-r[k], l.z, r[j + 2]);
        if (j + 3 > k + 1) r[j + 3] = fmaf(-r[k], l.w, r[j + 3]);
      }
    } else {
#pragma unroll
      for (int j = k + 2; j < kNB; ++j) r[j] = fmaf(-r[k], __shfl_sync(0xffffffffu, r[k], j), r[j]);
    }
  }
  if (!kShared)
#pragma unroll
    for (int c = 0; c < kNB; ++c) D[c * kNB + lane] = c <= lane ? r[c] : 0.f;
  rd[lane] = rdiag;
  return fail;
}

// x[j] -= L[j][k] xk for j > k; L's column k is read four entries at a time, the same for all lanes.
__device__ __forceinline__ void below_pivot(const float* L, int k, float xk, float (&x)[kNB]) {
#pragma unroll
  for (int j = (k + 1) & ~3; j < kNB; j += 4) {
    const float4 l = *reinterpret_cast<const float4*>(L + k * kNB + j);
    if (j > k) x[j] = fmaf(-l.x, xk, x[j]);
    if (j + 1 > k) x[j + 1] = fmaf(-l.y, xk, x[j + 1]);
    if (j + 2 > k) x[j + 2] = fmaf(-l.z, xk, x[j + 2]);
    if (j + 3 > k) x[j + 3] = fmaf(-l.w, xk, x[j + 3]);
  }
}

// Inv = L^-1 (column-major) for the factored diagonal block D with rd[k] = 1 / L_kk.  One warp.
// Column sweep: lane j solves L z = e_j; after step k, z[k] = Inv[k][j] is final.
template <bool kShared = true>
__device__ __noinline__ void warp_invert_factor(typename BlkPtr<kShared>::ro D, const float* __restrict__ rd,
                                                float* __restrict__ Inv) {
  const int lane = threadIdx.x & 31;
  float z[kNB];
#pragma unroll
  for (int i = 0; i < kNB; ++i) z[i] = i == lane ? 1.f : 0.f;
#pragma unroll
  for (int k = 0; k < kNB; ++k) {
    z[k] *= rd[k];
    below_pivot(D, k, z[k], z);
  }
#pragma unroll
  for (int i = 0; i < kNB; ++i) Inv[lane * kNB + i] = z[i];
}

// X L^T = A for one 32 x 32 block A (in place); lane owns a row.  L: factored diagonal block,
// rd[k] = 1 / L_kk.  Column k of X is final after step k and is eliminated from the later columns.
template <bool kShared = true>
__device__ __noinline__ void warp_solve_panel(typename BlkPtr<kShared>::rw A, typename BlkPtr<kShared>::ro L,
                                              const float* __restrict__ rd) {
  const int lane = threadIdx.x & 31;
  float a[kNB];
#pragma unroll
  for (int c = 0; c < kNB; ++c) a[c] = A[c * kNB + lane];
#pragma unroll
  for (int k = 0; k < kNB; ++k) {
    a[k] *= rd[k];
    below_pivot(L, k, a[k], a);
  }
#pragma unroll
  for (int c = 0; c < kNB; ++c) A[c * kNB + lane] = a[c];
}

// C -= A * Bm^T for 32 x 32 blocks (all column-major); lane computes a 4 x 8 sub-tile.
template <bool kShared>
__device__ __noinline__ void warp_rank32_update(typename BlkPtr<kShared>::rw C, typename BlkPtr<kShared>::ro A,
                                                typename BlkPtr<kShared>::ro Bm) {
  const int lane = threadIdx.x & 31, r0 = (lane & 7) * 4, c0 = (lane >> 3) * 8;
  float4 acc[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) acc[c] = *reinterpret_cast<const float4*>(C + (c0 + c) * kNB + r0);
#pragma unroll 8
  for (int p = 0; p < kNB; ++p) {
    const float4 a = *reinterpret_cast<const float4*>(A + p * kNB + r0);
    const float4 b0 = *reinterpret_cast<const float4*>(Bm + p * kNB + c0);
    const float4 b1 = *reinterpret_cast<const float4*>(Bm + p * kNB + c0 + 4);
    const float b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      acc[c].x = fmaf(-a.x, b[c], acc[c].x);
      acc[c].y = fmaf(-a.y, b[c], acc[c].y);
      acc[c].z = fmaf(-a.z, b[c], acc[c].z);
      acc[c].w = fmaf(-a.w, b[c], acc[c].w);
    }
  }
#pragma unroll
  for (int c = 0; c < 8; ++c) *reinterpret_cast<float4*>(C + (c0 + c) * kNB + r0) = acc[c];
}

// Solves L L^T x = v in place (v in shared memory, nb*32 entries, written by all warps in turn) with the blocked factor.
template <bool kShared = true>
__device__ __noinline__ void block_cholesky_solve(typename BlkPtr<kShared>::ro Lb, const float* __restrict__ InvD,
                                                  float* v, int nb) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  // forward: L y = v
  for (int J = 0; J < nb; ++J) {
    if (warp == 0) {
      const float* Inv = InvD + J * kBlk;
      float acc0 = 0.f, acc1 = 0.f;
#pragma unroll
      for (int k = 0; k < kNB; k += 2) {
        acc0 = fmaf(Inv[k * kNB + lane], v[J * kNB + k], acc0);
        acc1 = fmaf(Inv[(k + 1) * kNB + lane], v[J * kNB + k + 1], acc1);
      }
      __syncwarp();
      v[J * kNB + lane] = acc0 + acc1;
    }
    __syncthreads();
    for (int I = J + 1 + warp; I < nb; I += nwarps) {
      const float* L = Lb + blk_slot(I, J) * kBlk;
      float acc0 = v[I * kNB + lane], acc1 = 0.f;
#pragma unroll
      for (int p = 0; p < kNB; p += 2) {
        acc0 = fmaf(-L[p * kNB + lane], v[J * kNB + p], acc0);
        acc1 = fmaf(-L[(p + 1) * kNB + lane], v[J * kNB + p + 1], acc1);
      }
      v[I * kNB + lane] = acc0 + acc1;
    }
    __syncthreads();
  }
  // backward: L^T x = y; lane owns a row of the block, column sums by recursive halving
  for (int J = nb - 1; J >= 0; --J) {
    if (warp == 0) {
      const float* Inv = InvD + J * kBlk;
      const float yj = v[J * kNB + lane];
      float r[kNB];
#pragma unroll
      for (int i = 0; i < kNB; ++i) r[i] = Inv[i * kNB + lane] * yj;  // Inv[lane][i] y_lane
      v[J * kNB + lane] = warp_column_sums(r);                        // x_i = sum_k Inv[k][i] y_k
    }
    __syncthreads();
    for (int I = warp; I < J; I += nwarps) {
      const float* L = Lb + blk_slot(J, I) * kBlk;  // y_I -= L_JI^T x_J
      const float xj = v[J * kNB + lane];
      float r[kNB];
#pragma unroll
      for (int i = 0; i < kNB; ++i) r[i] = L[i * kNB + lane] * xj;
      v[I * kNB + lane] -= warp_column_sums(r);
    }
    __syncthreads();
  }
}

// Interacting variant, (K + lambda I) c = A: blocked Cholesky of the lower block triangle held at Lb (nb(nb+1)/2
// blocks; shared memory, or a workspace without kShared), the inverse diagonal factors at InvD, then the solve and up to
// two refinement rounds.  Called by every thread of a CTA of kThr; `layer` tags a failed pivot in *info.
template <int kThr = kSolveThreads, bool kShared = true>
__device__ __forceinline__ void interacting_solve(const TransformParams& P, float* Lb, float* InvD,
                                                  float* vec, double* sol, float* rdiag, double& s_trace, double& s_res,
                                                  int& s_fail, int layer) {
  const int B = P.B, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = kThr / 32;
  const float* __restrict__ K = P.K;
  const int nb = (B + kNB - 1) / kNB, Bp = nb * kNB;
  __shared__ int s_taken[2];  // trailing blocks of a column that warps have taken
  if (tid == 0) s_fail = s_taken[0] = s_taken[1] = 0;
  const bool vec4 = rows_in_float4(K, B);
  // load the lower block triangle.  K is symmetric, so row j of K read along i, from the block of the diagonal on, gives column j
  // of the blocks; a warp takes four rows at a time (float4 loads, eight in flight per lane, where rows are made of them).
  for (int j0 = warp * 4; j0 < B; j0 += nwarps * 4) {  // four columns of one block column
    const int J = j0 / kNB, first = J * kNB;
    if (vec4) {
      for (int i0 = first + lane * 4; i0 < B; i0 += 256) {
        float4 v[4][2];
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
          for (int h = 0; h < 2; ++h)
            v[u][h] = i0 + 128 * h < B ? __ldg(reinterpret_cast<const float4*>(K + (size_t)(j0 + u) * B + i0 + 128 * h)) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int i = i0 + 128 * h, j = j0 + u;
            if (i >= B) continue;
            float4 w = v[u][h];
            if (i == j) w.x += P.lambda;
            if (i + 1 == j) w.y += P.lambda;
            if (i + 2 == j) w.z += P.lambda;
            if (i + 3 == j) w.w += P.lambda;
            *reinterpret_cast<float4*>(Lb + blk_slot(i / kNB, J) * kBlk + (j % kNB) * kNB + (i % kNB)) = w;
          }
      }
    } else {
      for (int i = first + lane; i < B; i += 32)
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int j = j0 + u;
          if (j < B) Lb[blk_slot(i / kNB, J) * kBlk + (j % kNB) * kNB + (i % kNB)] = __ldg(K + (size_t)j * B + i) + (i == j ? P.lambda : 0.f);
        }
    }
  }
  // identity padding of the last block row / column
  for (int e = tid; e < (Bp - B) * Bp; e += kThr) {
    const int i = B + e / Bp, j = e % Bp;  // rows B..Bp-1, all columns j <= i
    if (j <= i || j / kNB == i / kNB)
      Lb[blk_slot(i / kNB, j / kNB) * kBlk + (j % kNB) * kNB + (i % kNB)] = i == j ? 1.f : 0.f;
  }
  __syncthreads();
  if (warp == 0) {
    const int f = warp_factor_diag<kShared>(Lb, rdiag);
    if (f != 0 && lane == 0) s_fail = f;
  }
  __syncthreads();
  for (int J = 0; J < nb && !s_fail; ++J) {
    const float* Ljj = Lb + blk_slot(J, J) * kBlk;
    if (tid == 0) s_taken[(J + 1) & 1] = 0;
    // panel: blocks (I, J) below the diagonal on warps 0 .. nwarps-2; the last warp inverts L_JJ
    if (warp == nwarps - 1) warp_invert_factor<kShared>(Ljj, rdiag + J * kNB, InvD + J * kBlk);
    else
      for (int I = J + 1 + warp; I < nb; I += nwarps - 1) warp_solve_panel<kShared>(Lb + blk_slot(I, J) * kBlk, Ljj, rdiag + J * kNB);
    __syncthreads();
    // trailing blocks (I, Kc) with I >= Kc > J; t = a(a+1)/2 + rem -> I = J+1+a, Kc = J+1+rem.
    // t = 0 is the next diagonal block: all warps update it together, then warp 0 factors it while the
    // others work through the rest
    const int m = nb - 1 - J, ntrail = m * (m + 1) / 2;
    if (m > 0) {
      // all warps: rank-32 update of the next diagonal block, kNB / nwarps columns each (lane = row)
      float* Dn = Lb + blk_slot(J + 1, J + 1) * kBlk;
      const float* Pn = Lb + blk_slot(J + 1, J) * kBlk;
      constexpr int kColsPerWarp = kNB / (kThr / 32);
      float acc[kColsPerWarp];
#pragma unroll
      for (int c = 0; c < kColsPerWarp; ++c) acc[c] = Dn[(warp * kColsPerWarp + c) * kNB + lane];
#pragma unroll 8
      for (int p = 0; p < kNB; ++p) {
        const float a = Pn[p * kNB + lane];
#pragma unroll
        for (int c = 0; c < kColsPerWarp; ++c) acc[c] = fmaf(-a, Pn[p * kNB + warp * kColsPerWarp + c], acc[c]);
      }
#pragma unroll
      for (int c = 0; c < kColsPerWarp; ++c) Dn[(warp * kColsPerWarp + c) * kNB + lane] = acc[c];
      __syncthreads();
      if (warp == 0) {
        const int f = warp_factor_diag<kShared>(Dn, rdiag + (J + 1) * kNB);
        if (f != 0 && lane == 0) s_fail = (J + 1) * kNB + f;
      }
      // The other blocks, whoever is free.  Warps 4, 8, .. share warp 0's scheduler and stay away: its factorisation is the serial
      // chain, and took 16.5 thousand clocks of the first column of 256 sequences among fifteen updating warps, 5.4 alone.  Not where the
      // updates are the longer (more than 64 blocks, which only the solve by one CTA above 256 sequences has: 1024 of them 2302 / 2182 us).
      if ((!kShared && ntrail > 64) || warp == 0 || (warp & 3) != 0) {
        while (true) {
          int t = 0;
          if (lane == 0) t = 1 + atomicAdd(&s_taken[J & 1], 1);
          t = __shfl_sync(0xffffffffu, t, 0);
          if (t >= ntrail) break;
          int a = 0, rem = t;
          while (rem > a) { rem -= a + 1; ++a; }
          const int I = J + 1 + a, Kc = J + 1 + rem;
          warp_rank32_update<kShared>(Lb + blk_slot(I, Kc) * kBlk, Lb + blk_slot(I, J) * kBlk, Lb + blk_slot(Kc, J) * kBlk);
        }
      }
    }
    __syncthreads();
  }
  __syncthreads();
  if (s_fail) {
    if (tid == 0) atomicCAS(P.info, 0, s_fail + (layer << 16));
    for (int i = tid; i < B; i += kThr) P.coeffs[i] = 0.f;
    return;
  }
  // solve, then refinement rounds with a float64 residual while it is above float32 round-off
  double anorm2 = 0.0;
  for (int i = tid; i < Bp; i += kThr) {
    const float a = i < B ? P.A[i] : 0.f;
    vec[i] = a;
    sol[i] = 0.0;
    anorm2 += (double)a * a;
  }
  anorm2 = warp_sum(anorm2);
  if (tid == 0) { s_trace = 0.0; s_res = 0.0; }
  __syncthreads();
  if (lane == 0) atomicAdd(&s_trace, anorm2);
  __syncthreads();
  anorm2 = s_trace;
  for (int round = 0; round < 3; ++round) {
    block_cholesky_solve<kShared>(Lb, InvD, vec, nb);
    for (int i = tid; i < Bp; i += kThr) sol[i] += (double)vec[i];
    __syncthreads();
    if (round == 2) break;
    double rn2 = 0.0;
    for (int i0 = warp * 4; i0 < B; i0 += nwarps * 4) {  // four rows per warp pass: independent loads
      double acc[4] = {0.0, 0.0, 0.0, 0.0};
      if (vec4) {
        for (int j0 = lane * 4; j0 < B; j0 += 256) {  // two float4 per lane and row in flight
          float4 kv[4][2];
#pragma unroll
          for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const int j = j0 + h * 128;
              kv[u][h] = (i0 + u < B && j < B) ? __ldg(reinterpret_cast<const float4*>(K + (size_t)(i0 + u) * B + j))
                                              : make_float4(0.f, 0.f, 0.f, 0.f);
            }
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int j = j0 + h * 128;
            if (j >= B) continue;
            const double s0 = sol[j], s1 = sol[j + 1], s2 = sol[j + 2], s3 = sol[j + 3];
#pragma unroll
            for (int u = 0; u < 4; ++u)
              acc[u] += (double)kv[u][h].x * s0 + (double)kv[u][h].y * s1 + (double)kv[u][h].z * s2 +
                        (double)kv[u][h].w * s3;
          }
        }
      } else {
        for (int j = lane; j < B; j += 32) {
          const double sj = sol[j];
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (i0 + u < B) acc[u] += (double)K[(size_t)(i0 + u) * B + j] * sj;
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const double a = warp_sum(acc[u]);
        if (lane == 0 && i0 + u < B) {
          const double r = (double)P.A[i0 + u] - a - (double)P.lambda * sol[i0 + u];
          vec[i0 + u] = (float)r;
          rn2 += r * r;
        }
      }
    }
    if (lane == 0) atomicAdd(&s_res, rn2);
    __syncthreads();
    const bool done = s_res <= 1e-14 * anorm2;  // relative residual below 1e-7
    __syncthreads();
    if (tid == 0) s_res = 0.0;
    if (done) break;
  }
  for (int i = tid; i < B; i += kThr) P.coeffs[i] = (float)sol[i];
}

// Dynamic shared memory of a CTA that runs interacting_solve, and its layout.
struct SolveSmem {
  float* Lb;     // nb(nb+1)/2 blocks
  float* InvD;   // nb inverse diagonal factors
  float* vec;    // Bp floats
  double* sol;   // Bp doubles (8-byte aligned: all counts even)
  float* rdiag;  // Bp floats: 1 / L_kk
};
__device__ __forceinline__ SolveSmem solve_smem(unsigned char* raw, int B) {
  const int nb = (B + kNB - 1) / kNB, Bp = nb * kNB;
  SolveSmem m;
  m.Lb = reinterpret_cast<float*>(raw);
  m.InvD = m.Lb + (size_t)(nb * (nb + 1) / 2) * kBlk;
  m.vec = m.InvD + (size_t)nb * kBlk;
  m.sol = reinterpret_cast<double*>(m.vec + Bp);
  m.rdiag = reinterpret_cast<float*>(m.sol + Bp);
  return m;
}
inline size_t solve_smem_bytes(int B) {
  const size_t nb = (size_t)(B + kNB - 1) / kNB;
  return sizeof(float) * ((nb * (nb + 1) / 2 + nb) * kBlk + 2 * nb * kNB) + sizeof(double) * nb * kNB;
}

}  // namespace

}  // namespace isopo
