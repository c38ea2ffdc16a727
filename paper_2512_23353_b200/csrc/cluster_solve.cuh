// Interacting solve (K + lambda I) c = A for 257 to 1024 sequences by one cluster of sixteen CTAs: blocked Cholesky
// (float32, 32 x 32 blocks), blocked triangular solves, up to two refinement rounds with float64 residuals from the
// float32 K, stopped once the relative residual is below 1e-7: the method of interacting_solve.cuh, spread over 16 SMs.
//
// Block rows of the matrix are dealt to the CTAs in a snake (0 .. C-1, C-1 .. 0, ..), so that every CTA has about the
// same number of blocks, and stay in its shared memory from K to L.  Block column J:
//   panel      L_IJ = A_IJ Inv_J^T for the own rows, Inv_J the inverse of the diagonal factor; published in the
//              workspace, which stays in the L2
//   barrier 1  every panel block is visible
//   trailing   A_IK -= L_IJ L_KJ^T for the own rows, a warp per block; beside it the owner of row J + 1, which has updated
//              its diagonal block first, factors and inverts it with one warp and publishes Inv_{J+1}
//   barrier 2  Inv_{J+1} is visible
// The right-hand side rides along, so the forward substitution of the first solve costs nothing.  In the other
// substitutions the owner of a block row computes its 32 unknowns and sends them to everybody (st.async, one transaction
// barrier per block row); the owners of the remaining rows have the block they need in registers before the unknowns
// arrive.
//
// Bound by latency: per block column two cluster barriers and the serial chain panel - diagonal update - factor - inverse.
// Measured against one CTA with the factor in the workspace: 512 sequences 145 against 398 us, 1024: 340 against 2207 us.  A
// cluster of eight with the panels in shared memory, tried for 129 to 256 sequences, took 53 to 82 us where the one CTA
// of interacting_solve.cuh takes 53 to 90 (192: 63 against 61): not kept.
#pragma once

#include "interacting_solve.cuh"
#include "tc_common.cuh"

namespace isopo {

namespace {

constexpr int kClThreads = 512;
constexpr int kClWarps = kClThreads / 32;

__device__ __forceinline__ void cl_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cl_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void st_cluster_f32(uint32_t addr, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ void st_cluster_f64(uint32_t addr, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(addr), "d"(v) : "memory");
}
__device__ __forceinline__ void st_async_f32x4(uint32_t addr, const float4& v, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(addr),
               "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"(bar)
               : "memory");
}

constexpr int kMaxOwn = 2;  // block rows of a CTA: 32 / 16

// Fixed part of the dynamic shared memory; the own blocks follow.
struct ClSmem {
  uint64_t bar[2][32];      // unknowns of block row J: forward, backward
  float inv[2][kBlk];       // Inv_J, alternating
  float inv_own[kMaxOwn][kBlk];
  float rhs[2][kNB];        // right-hand side of block row J, with Inv_J
  float own_rhs[kMaxOwn][kNB];
  float y[1024], x[1024];   // solution of the forward / backward substitution
  double sol[1024];
  double part[16];          // squared residual of every CTA
  double red[kClWarps];
  float z[kMaxOwn][kNB];
  float rdiag[kNB];
  int fail[2];
  int abort_flag;
};
// read and written 16 bytes at a time
static_assert(offsetof(ClSmem, inv) % 16 == 0 && offsetof(ClSmem, inv_own) % 16 == 0 && offsetof(ClSmem, y) % 16 == 0 &&
              offsetof(ClSmem, x) % 16 == 0 && offsetof(ClSmem, z) % 16 == 0, "alignment");
__host__ __device__ inline int cl_own_blocks(int nb, int C) {  // most blocks of one CTA
  return nb <= C ? nb : 2 * C + 1;
}
template <int kC>
inline size_t cl_smem_bytes(int B) {
  const int nb = (B + kNB - 1) / kNB;
  return sizeof(ClSmem) + sizeof(float) * kBlk * (size_t)cl_own_blocks(nb, kC) + 128;
}

// P: K, A, B, lambda, coeffs, info.  Lg: nb (nb + 1) / 2 blocks of workspace: L below the diagonal, Inv on it.
template <int kC>
__device__ __forceinline__ void cluster_solve(const TransformParams& P, float* Lg, unsigned char* smem_raw, int layer) {
  ClSmem& S = *reinterpret_cast<ClSmem*>(smem_raw);
  float* blocks = reinterpret_cast<float*>(smem_raw + ((sizeof(ClSmem) + 127) & ~size_t(127)));
  const int B = P.B, nb = (B + kNB - 1) / kNB, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = (int)tc::cluster_ctarank();
  const float* __restrict__ K = P.K;
  const int rows[kMaxOwn] = {rank, 2 * kC - 1 - rank};           // own block rows; those >= nb do not exist
  auto blk = [&](int l, int J) { return blocks + (size_t)((l == 0 ? 0 : rank + 1) + J) * kBlk; };
  auto at = [&](const void* p, int cta) { return tc::map_to_cta(tc::smem_u32(p), (uint32_t)cta); };
  const uint32_t bar0 = tc::smem_u32(&S.bar[0][0]);

  // ---- load the own block rows (K is symmetric: row j read along i gives column j of the blocks) ----
#pragma unroll
  for (int l = 0; l < kMaxOwn; ++l) {
    const int I = rows[l];
    if (I >= nb) continue;
    const int i = I * kNB + lane;
#pragma unroll 8
    for (int c = warp; c < (I + 1) * kNB; c += kClWarps) {  // column c of the block row
      float v = i == c ? 1.f : 0.f;                         // identity padding
      if (i < B && c < B) v = __ldg(K + (size_t)c * B + i) + (i == c ? P.lambda : 0.f);
      blk(l, c / kNB)[(c % kNB) * kNB + lane] = v;
    }
    if (warp == 0) S.own_rhs[l][lane] = i < B ? P.A[i] : 0.f;
  }
  double anorm2 = 0.0;
  for (int i = tid; i < B; i += kClThreads) anorm2 += (double)P.A[i] * P.A[i];
  anorm2 = warp_sum(anorm2);
  if (lane == 0) S.red[warp] = anorm2;
  if (tid == 0) {
    S.abort_flag = 0;
    S.fail[0] = S.fail[1] = 0;
    for (int k = 0; k < 64; ++k) tc::mbar_init(bar0 + 8 * k, 1);
    tc::fence_barrier_init();
  }
  for (int i = tid; i < 1024; i += kClThreads) S.sol[i] = 0.0;
  __syncthreads();
  anorm2 = 0.0;
  for (int w = 0; w < kClWarps; ++w) anorm2 += S.red[w];
  cl_arrive();
  cl_wait();  // everybody runs and its barriers exist

  // Factors and inverts the diagonal block of own row l and publishes the inverse, the right-hand side and whether a pivot
  // failed.  One warp of the owner.
  auto factor = [&](int l, int J) {
    const int f = warp_factor_diag<false>(blk(l, J), S.rdiag);
    __syncwarp();
    warp_invert_factor(blk(l, J), S.rdiag, S.inv_own[l]);
    __syncwarp();
    const int b = J & 1;
    const float4* src = reinterpret_cast<const float4*>(S.inv_own[l]);
#pragma unroll
    for (int u = 0; u < kBlk / 128; ++u) {
      reinterpret_cast<float4*>(Lg + (size_t)blk_slot(J, J) * kBlk)[u * 32 + lane] = src[u * 32 + lane];
    }
    const float a = S.own_rhs[l][lane];
#pragma unroll
    for (int t = 0; t < kC; ++t) st_cluster_f32(at(&S.rhs[b][lane], t), a);
    if (lane < kC) tc::st_cluster_u32(at(&S.fail[b], lane), (uint32_t)(f ? J * kNB + f : 0));
  };
  auto fetch_inv = [&](int J) {
    if (tid < kBlk / 4)
      reinterpret_cast<float4*>(S.inv[J & 1])[tid] = __ldcg(reinterpret_cast<const float4*>(Lg + (size_t)blk_slot(J, J) * kBlk) + tid);
  };
  if (rank == 0 && warp == 0) factor(0, 0);
  cl_arrive();
  cl_wait();

  // ---- factorisation, forward substitution of the right-hand side ----
  int failed = 0;
  for (int J = 0; J < nb; ++J) {
    fetch_inv(J);
    failed = S.fail[J & 1];
    if (failed) break;  // the same in every thread of the cluster
    __syncthreads();
    const float* inv = S.inv[J & 1];
    // panel: two columns per warp, lane = row
    float acc[kMaxOwn][2] = {};
#pragma unroll
    for (int l = 0; l < kMaxOwn; ++l) {
      if (rows[l] <= J || rows[l] >= nb) continue;
      const float* A = blk(l, J);
#pragma unroll 8
      for (int k = 0; k < kNB; ++k) {
        const float a = A[k * kNB + lane];
        const float2 v = *reinterpret_cast<const float2*>(inv + k * kNB + 2 * warp);
        acc[l][0] = fmaf(a, v.x, acc[l][0]);
        acc[l][1] = fmaf(a, v.y, acc[l][1]);
      }
    }
    if (warp == kClWarps - 1) {
      float v = 0.f;
#pragma unroll 8
      for (int k = 0; k < kNB; ++k) v = fmaf(inv[k * kNB + lane], S.rhs[J & 1][k], v);
      S.y[J * kNB + lane] = v;
    }
    __syncthreads();
#pragma unroll
    for (int l = 0; l < kMaxOwn; ++l) {
      const int I = rows[l];
      if (I <= J || I >= nb) continue;
      float* A = blk(l, J);
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const int e = (2 * warp + c) * kNB + lane;
        A[e] = acc[l][c];
        Lg[(size_t)blk_slot(I, J) * kBlk + e] = acc[l][c];
      }
    }
    cl_arrive();
    __syncthreads();  // the own blocks of the panel and y_J are complete
    const int next = J + 1 < nb ? (rows[0] == J + 1 ? 0 : rows[1] == J + 1 ? 1 : -1) : -1;  // own row to factor next
    if (warp < kMaxOwn) {  // right-hand side of the own rows
      const int l = next >= 0 ? (warp == 0 ? next : 1 - next) : warp;
      if (rows[l] > J && rows[l] < nb) {
        const float* L = blk(l, J);
        float v = S.own_rhs[l][lane];
#pragma unroll 8
        for (int k = 0; k < kNB; ++k) v = fmaf(-L[k * kNB + lane], S.y[J * kNB + k], v);
        S.own_rhs[l][lane] = v;
      }
      __syncwarp();
    }
    if (next >= 0) {
      float* Dn = blk(next, J + 1);
      const float* Pn = blk(next, J);
      float d[2];
#pragma unroll
      for (int c = 0; c < 2; ++c) d[c] = Dn[(2 * warp + c) * kNB + lane];
#pragma unroll 8
      for (int k = 0; k < kNB; ++k) {
        const float a = Pn[k * kNB + lane];
        const float2 v = *reinterpret_cast<const float2*>(Pn + k * kNB + 2 * warp);
        d[0] = fmaf(-a, v.x, d[0]);
        d[1] = fmaf(-a, v.y, d[1]);
      }
#pragma unroll
      for (int c = 0; c < 2; ++c) Dn[(2 * warp + c) * kNB + lane] = d[c];
      __syncthreads();
      if (warp == 0) factor(next, J + 1);
    }
    cl_wait();  // every panel block is visible
    // trailing blocks of the own rows, one per warp at a time; warp 0 of the next owner is busy
    const int workers = next >= 0 ? kClWarps - 1 : kClWarps, me = next >= 0 ? warp - 1 : warp;
    if (me >= 0) {
      int first = 0;
#pragma unroll
      for (int l = 0; l < kMaxOwn; ++l) {
        const int I = rows[l];
        if (I <= J || I >= nb) continue;
        const int count = I - J - (l == next ? 1 : 0);  // columns J + 1 .. I, without the diagonal block done above
        int k = me - first % workers;
        if (k < 0) k += workers;
        for (; k < count; k += workers) {
          const int Kc = J + 1 + k;
          warp_rank32_update<false>(blk(l, Kc), blk(l, J), Lg + (size_t)blk_slot(Kc, J) * kBlk);
        }
        first += count;
      }
    }
    cl_arrive();
    cl_wait();  // the next inverse is visible, and nobody reads this panel any more
  }
  if (failed) {
    if (rank == 0) {
      if (tid == 0) atomicCAS(P.info, 0, failed + (layer << 16));
      for (int i = tid; i < B; i += kClThreads) P.coeffs[i] = 0.f;
    }
    return;
  }

  // ---- substitutions ----
  // Sends the 32 values v (one per lane) of block row J to everybody's dst and raises bar there.
  auto send = [&](float* scratch, float v, float* dst, uint32_t bar) {
    scratch[lane] = v;
    __syncwarp();
    const float4 q = *reinterpret_cast<const float4*>(scratch + 4 * (lane & 7));
#pragma unroll
    for (int t = 0; t < kC; t += 4) {
      const int cta = t + (lane >> 3);
      st_async_f32x4(at(dst + 4 * (lane & 7), cta), q, tc::map_to_cta(bar, (uint32_t)cta));
    }
    __syncwarp();
  };
  auto wait = [&](int set, int J, int round) {
    return tc::mbar_wait(bar0 + 8 * (32 * set + J), (uint32_t)round & 1u, &S.abort_flag, P.info, kIdTransform);
  };
  auto dot32 = [&](const float (&m)[kNB], const float* v) {  // v: shared memory, the same for all lanes
    float s[4] = {};
#pragma unroll
    for (int k = 0; k < kNB; k += 4) {
      const float4 q = *reinterpret_cast<const float4*>(v + k);
      s[0] = fmaf(m[k], q.x, s[0]); s[1] = fmaf(m[k + 1], q.y, s[1]);
      s[2] = fmaf(m[k + 2], q.z, s[2]); s[3] = fmaf(m[k + 3], q.w, s[3]);
    }
    return (s[0] + s[1]) + (s[2] + s[3]);
  };
  // row / column `lane` of a column-major block
  auto load_rows = [&](float (&m)[kNB], const float* p) {
#pragma unroll
    for (int k = 0; k < kNB; ++k) m[k] = p[k * kNB + lane];
  };
  auto load_cols = [&](float (&m)[kNB], const float* p) {
#pragma unroll
    for (int k = 0; k < kNB; k += 4) {
      const float4 q = *reinterpret_cast<const float4*>(p + lane * kNB + k);
      m[k] = q.x; m[k + 1] = q.y; m[k + 2] = q.z; m[k + 3] = q.w;
    }
  };

  for (int round = 0; round < 3; ++round) {
    if (tid < 64 && lane < nb) tc::mbar_arrive_expect_tx(bar0 + 8 * tid, kNB * 4);  // both sets, once a round
    __syncthreads();
    if (round > 0) {
      // L y = r, r in own_rhs
      if (warp < kMaxOwn && rows[warp] < nb) {
        const int I = rows[warp];
        float v = S.own_rhs[warp][lane], m[kNB];
        for (int J = 0; J < I; ++J) {
          load_rows(m, blk(warp, J));
          wait(0, J, round);
          v -= dot32(m, S.y + J * kNB);
        }
        load_rows(m, S.inv_own[warp]);
        S.z[warp][lane] = v;
        __syncwarp();
        v = dot32(m, S.z[warp]);
        __syncwarp();
        send(S.z[warp], v, S.y + I * kNB, bar0 + 8 * I);
      }
      if (warp == kMaxOwn && lane < nb) wait(0, lane, round);
      __syncthreads();
    } else if (warp < kMaxOwn && rows[warp] < nb) {  // y is there already: raise the forward barriers of this round all the same
      send(S.z[warp], S.y[rows[warp] * kNB + lane], S.y + rows[warp] * kNB, bar0 + 8 * rows[warp]);
    }
    // L^T x = y
    if (warp < kMaxOwn && rows[warp] < nb) {
      const int I = rows[warp];
      float v = S.y[I * kNB + lane], m[kNB];
      for (int J = nb - 1; J > I; --J) {
        load_cols(m, Lg + (size_t)blk_slot(J, I) * kBlk);
        wait(1, J, round);
        v -= dot32(m, S.x + J * kNB);
      }
      load_cols(m, S.inv_own[warp]);
      S.z[warp][lane] = v;
      __syncwarp();
      v = dot32(m, S.z[warp]);
      __syncwarp();
      send(S.z[warp], v, S.x + I * kNB, bar0 + 8 * (32 + I));
    }
    if (warp == kMaxOwn && lane < nb) { wait(1, lane, round); wait(0, lane, round); }
    __syncthreads();
    for (int i = tid; i < B; i += kClThreads) S.sol[i] += (double)S.x[i];
    __syncthreads();
    if (round == 2) break;
    // residual of the own rows, four per warp
    double rn2 = 0.0;
#pragma unroll 1
    for (int g = warp; g < kMaxOwn * 8; g += kClWarps) {
      const int l = g >> 3, r0 = (g & 7) * 4, I = l == 0 ? rows[0] : rows[1];
      if (I >= nb) continue;
      double acc[4] = {};
      if (rows_in_float4(K, B)) {
        for (int j = lane * 4; j < B; j += 128) {
          const double q0 = S.sol[j], q1 = S.sol[j + 1], q2 = S.sol[j + 2], q3 = S.sol[j + 3];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const float4 v = __ldg(reinterpret_cast<const float4*>(K + (size_t)min(I * kNB + r0 + u, B - 1) * B + j));
            acc[u] += (double)v.x * q0 + (double)v.y * q1 + (double)v.z * q2 + (double)v.w * q3;
          }
        }
      } else {
        for (int j = lane; j < B; j += 32) {
          const double q = S.sol[j];
#pragma unroll
          for (int u = 0; u < 4; ++u) acc[u] += (double)__ldg(K + (size_t)min(I * kNB + r0 + u, B - 1) * B + j) * q;
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const double a = warp_sum(acc[u]);
        const int i = I * kNB + r0 + u;
        const double r = i < B ? (double)P.A[i] - a - (double)P.lambda * S.sol[i] : 0.0;
        if (lane == 0) { S.own_rhs[l][r0 + u] = (float)r; rn2 += r * r; }
      }
    }
    if (lane == 0) S.red[warp] = rn2;
    __syncthreads();
    if (tid < kC) {
      double t = 0.0;
      for (int w = 0; w < kClWarps; ++w) t += S.red[w];
      st_cluster_f64(at(&S.part[rank], tid), t);
    }
    cl_arrive();
    cl_wait();
    rn2 = 0.0;
    for (int t = 0; t < kC; ++t) rn2 += S.part[t];
    if (rn2 <= 1e-14 * anorm2) break;  // relative residual below 1e-7; the same in every thread of the cluster
    cl_arrive();
    cl_wait();  // nobody overwrites a part that is still read
  }
  if (rank == 0)
    for (int i = tid; i < B; i += kClThreads) P.coeffs[i] = (float)S.sol[i];
  if (S.abort_flag) __nanosleep(100000);
  cl_arrive();
  cl_wait();  // nobody leaves while another CTA may still send to it
}

}  // namespace

}  // namespace isopo
