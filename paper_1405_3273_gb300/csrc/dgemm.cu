// FP64 building blocks: a strided, doubly-batched GEMM on the CUDA cores and a
// one-cluster Gauss-Jordan inverse for the (symmetric positive-definite) overlap.
//
// The GEMM computes, for every batch index (b0, b1),
//   C[b] = alpha * A[b] B[b] + beta_c * C[b]
// with arbitrary row/column/batch strides, so that every single-index
// contraction of a 4-index tensor by an N x N matrix maps onto it without
// copies.  64x64 output tile per CTA, 256 threads with 4x4 outputs each,
// K consumed in slabs of 16 staged through shared memory.  FP64 FMA on
// GB300 is the bound, not memory.
#include <algorithm>
#include <utility>

#include <cooperative_groups.h>

#include "gf2_internal.cuh"

namespace {

namespace cg = cooperative_groups;

constexpr int TM = 64, TN = 64, TK = 16;

__global__ void __launch_bounds__(256) dgemm_kernel(Dgemm g, int tiles_m, int tiles_n) {
  __shared__ double As[TK][TM + 1];
  __shared__ double Bs[TK][TN + 1];
  const int tile = blockIdx.x;
  const int ks = g.split_k > 1 ? g.split_k : 1;
  const int kpart = tile % ks;
  const int t = tile / ks;
  const int tm = t / tiles_n, tn = t % tiles_n;
  const int b0 = blockIdx.y, b1 = blockIdx.z;
  const double *A = g.A + b0 * g.a_b0 + b1 * g.a_b1;
  const double *B = g.B + b0 * g.b_b0 + b1 * g.b_b1;
  double *C = g.C + b0 * g.c_b0 + b1 * g.c_b1;

  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  const int row0 = tm * TM, col0 = tn * TN;
  double acc[4][4] = {};

  long long kchunk = ((long long)g.K + ks - 1) / ks;
  kchunk = ((kchunk + TK - 1) / TK) * TK;
  const long long kbeg = kpart * kchunk;
  const long long kend = min((long long)g.K, kbeg + kchunk);

  for (long long k0 = kbeg; k0 < kend; k0 += TK) {
    // stage A[row0:+64, k0:+16] and B[k0:+16, col0:+64]
    for (int e = threadIdx.x; e < TM * TK; e += 256) {
      int r = e / TK, kk = e % TK;
      long long gr = row0 + r, gk = k0 + kk;
      As[kk][r] = (gr < g.M && gk < kend) ? A[gr * g.a_rs + gk * g.a_cs] : 0.0;
    }
    for (int e = threadIdx.x; e < TK * TN; e += 256) {
      int kk = e / TN, c = e % TN;
      long long gc = col0 + c, gk = k0 + kk;
      Bs[kk][c] = (gc < g.N && gk < kend) ? B[gk * g.b_rs + gc * g.b_cs] : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < TK; ++kk) {
      double a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = As[kk][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = Bs[kk][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    long long gr = row0 + ty + 16 * i;
    if (gr >= g.M) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      long long gc = col0 + tx + 16 * j;
      if (gc >= g.N) continue;
      double *c = C + gr * g.c_rs + gc * g.c_cs;
      if (ks > 1) {
        atomicAdd(c, g.alpha * acc[i][j]);
      } else {
        double prev = g.beta_c != 0.0 ? g.beta_c * (*c) : 0.0;
        *c = g.alpha * acc[i][j] + prev;
      }
    }
  }
}

// The same product for matrices too small to fill the chip with 64 x 64 tiles: an
// SM does two FP64 multiply-adds per clock, so a 64 x 64 x 64 product on one SM takes
// 68 us whatever its latencies.  8 x 8 outputs per CTA: 64 SMs share that product.
// Every output is the same chain of multiply-adds as above (K ascending), bit for
// bit: what is built on these products (the Loewdin basis of the split path) does
// not depend on which kernel ran.
constexpr int SM_T = 8, SM_K = 64;
__global__ void __launch_bounds__(SM_T *SM_T) dgemm_small_kernel(Dgemm g, int tiles_n) {
  __shared__ double As[SM_T][SM_K + 1], Bs[SM_K][SM_T + 1];
  const int tm = blockIdx.x / tiles_n, tn = blockIdx.x % tiles_n;
  const double *A = g.A + blockIdx.y * g.a_b0 + blockIdx.z * g.a_b1;
  const double *B = g.B + blockIdx.y * g.b_b0 + blockIdx.z * g.b_b1;
  double *C = g.C + blockIdx.y * g.c_b0 + blockIdx.z * g.c_b1;
  const int r = threadIdx.x / SM_T, c = threadIdx.x % SM_T, row0 = tm * SM_T, col0 = tn * SM_T;
  double acc = 0.0;
  for (int k0 = 0; k0 < g.K; k0 += SM_K) {
#pragma unroll
    for (int q = 0; q < SM_T; ++q) {
      const int ka = threadIdx.x, kb = q * SM_T + r;
      As[q][ka] = (row0 + q < g.M && k0 + ka < g.K) ? A[(row0 + q) * g.a_rs + (k0 + ka) * g.a_cs] : 0.0;
      Bs[kb][c] = (col0 + c < g.N && k0 + kb < g.K) ? B[(k0 + kb) * g.b_rs + (col0 + c) * g.b_cs] : 0.0;
    }
    __syncthreads();
    const int ke = min(SM_K, g.K - k0);
#pragma unroll 8
    for (int k = 0; k < ke; ++k) acc = fma(As[r][k], Bs[k][c], acc);
    __syncthreads();
  }
  if (row0 + r < g.M && col0 + c < g.N) {
    double *o = C + (row0 + r) * g.c_rs + (col0 + c) * g.c_cs;
    const double prev = g.beta_c != 0.0 ? g.beta_c * (*o) : 0.0;
    *o = g.alpha * acc + prev;
  }
}

// Gauss-Jordan inversion of an SPD matrix (no pivoting needed) by a cluster of
// eight CTAs, each holding n / 8 columns in registers.  Pivot k: the owner of
// column k sends it and the reciprocal pivot to every CTA's shared memory, one
// cluster barrier, every CTA updates its columns; the two buffers alternate, so
// that barrier is the only one per pivot.  One more comes before the first pivot (a
// CTA's shared memory may be written only once it has started; its arrival and its
// wait enclose the loads of A) and one after the last.  One SM alone is bound by its two FP64 multiply-adds
// per clock (n^3 of them) and by the division that all its threads repeated: 235 us
// at n = 64, 121 us here, of which the reciprocals are most.
constexpr int kInvCtas = 8, kInvThreads = 256;
constexpr int kInvPer = GF2_MAX_N * ((GF2_MAX_N + kInvCtas - 1) / kInvCtas) / kInvThreads;
__global__ void __cluster_dims__(kInvCtas, 1, 1) __launch_bounds__(kInvThreads)
    inverse_spd_kernel(const double *A, double *Ainv, int n) {
  // a launch that asks for it (the energy sum, which needs nothing from here) may
  // start now, beside these eight CTAs
  cudaTriggerProgrammaticLaunchCompletion();
  __shared__ double col[2][GF2_MAX_N], row[2][GF2_MAX_N / kInvCtas], piv[2];
  cg::cluster_group cluster = cg::this_cluster();
  const int W = (n + kInvCtas - 1) / kInvCtas, j0 = (int)cluster.block_rank() * W, w = max(0, min(W, n - j0));
  double a[kInvPer];
  auto started = cluster.barrier_arrive();
#pragma unroll
  for (int r = 0; r < kInvPer; ++r) {
    const int e = threadIdx.x + r * kInvThreads;
    a[r] = e < n * w ? A[(e / w) * n + j0 + e % w] : 0.0;
  }
  cluster.barrier_wait(std::move(started));
  for (int k = 0; k < n; ++k) {
    const int buf = k & 1;
#pragma unroll
    for (int r = 0; r < kInvPer; ++r) {
      const int e = threadIdx.x + r * kInvThreads;
      if (e >= n * w) break;
      const int i = e / w, jl = e % w, j = j0 + jl;
      if (i == k) row[buf][jl] = a[r];
      if (j == k) {
        const double p = i == k ? 1.0 / a[r] : 0.0;
        for (int d = 0; d < kInvCtas; ++d) {
          cluster.map_shared_rank(&col[buf][0], d)[i] = a[r];
          if (i == k) *cluster.map_shared_rank(&piv[buf], d) = p;
        }
      }
    }
    cluster.sync();
    const double p = piv[buf];
#pragma unroll
    for (int r = 0; r < kInvPer; ++r) {
      const int e = threadIdx.x + r * kInvThreads;
      if (e >= n * w) break;
      const int i = e / w, jl = e % w, j = j0 + jl;
      const double rj = j == k ? p : row[buf][jl] * p;
      if (i == k) a[r] = rj;
      else if (j == k) a[r] = -col[buf][i] * p;
      else a[r] -= col[buf][i] * rj;
    }
  }
  cluster.sync();  // no CTA ends while another may still write into it
#pragma unroll
  for (int r = 0; r < kInvPer; ++r) {
    const int e = threadIdx.x + r * kInvThreads;
    if (e < n * w) Ainv[(e / w) * n + j0 + e % w] = a[r];
  }
}

}  // namespace

gf2_status gf2_dgemm(gf2_ctx *ctx, const Dgemm &g) {
  if (g.M <= 0 || g.N <= 0 || g.K <= 0 || g.nb0 <= 0 || g.nb1 <= 0) return GF2_OK;
  if (g.nb0 > 65535 || g.nb1 > 65535) return gf2_fail(ctx, GF2_ERR_UNSUPPORTED, "dgemm batch too large");
  const int tiles_m = (g.M + TM - 1) / TM, tiles_n = (g.N + TN - 1) / TN;
  const int ks = g.split_k > 1 ? g.split_k : 1;
  dim3 grid(tiles_m * tiles_n * ks, g.nb0, g.nb1);
  // 64 x 64 tiles where they give every SM one, the small ones below that
  if (ks == 1 && (long long)tiles_m * tiles_n * g.nb0 * g.nb1 < ctx->num_sms) {
    const int sm = (g.M + SM_T - 1) / SM_T, sn = (g.N + SM_T - 1) / SM_T;
    GF2_PROF(ctx, GF2_K_DGEMM, (dgemm_small_kernel<<<dim3(sm * sn, g.nb0, g.nb1), SM_T * SM_T, 0, ctx->stream>>>(g, sn)));
    GF2_CK_LAUNCH(ctx, "dgemm_small_kernel");
    return GF2_OK;
  }
  GF2_PROF(ctx, GF2_K_DGEMM, (dgemm_kernel<<<grid, 256, 0, ctx->stream>>>(g, tiles_m, tiles_n)));
  GF2_CK_LAUNCH(ctx, "dgemm_kernel");
  return GF2_OK;
}

gf2_status gf2_inverse_spd(gf2_ctx *ctx, const double *d_A, double *d_Ainv) {
  const int n = ctx->N;
  inverse_spd_kernel<<<kInvCtas, kInvThreads, 0, ctx->stream>>>(d_A, d_Ainv, n);
  GF2_CK_LAUNCH(ctx, "inverse_spd_kernel");
  return GF2_OK;
}
