// FP64 batched GEMM for the propagator builder and the plain FP64 apply.
//   C[b](m, n) = alpha * sum_k A[b](m, k) * B[b](k, n) + beta * C[b](m, n)
// Row-major operands. transB = 1 reads B(k, n) from B[n * ldb + k] (B stored N x K).
// An optional row index maps A row m and C row m to rowidx[m] (gathered rows), which the
// step uses to apply one class propagator to the tiles of that class.
// GB300 runs FP64 at about 1.2 TFLOP/s (two DFMA per clock per SM), so this kernel is
// bound by the FP64 pipe: 64 x 64 CTA tile, 4 x 4 outputs per thread, 16-deep K slabs
// staged in shared memory; loads are guarded so any M, N, K works.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace lem {

struct DgemmArgs {
  int M, N, K;
  const double* A; int64_t lda; int64_t sA;
  const double* B; int64_t ldb; int64_t sB; int transB;
  double* C; int64_t ldc; int64_t sC;
  double alpha, beta;
  const int32_t* rowidx;  // optional (nullptr): A/C row m -> rowidx[m]
};

constexpr int DG_BM = 64, DG_BN = 64, DG_BK = 16;

static __global__ void __launch_bounds__(256) dgemm_kernel(DgemmArgs g) {
  __shared__ double As[DG_BK][DG_BM + 1];
  __shared__ double Bs[DG_BK][DG_BN + 1];
  const int b = blockIdx.z;
  const double* A = g.A + b * g.sA;
  const double* B = g.B + b * g.sB;
  double* C = g.C + b * g.sC;
  const int m0 = blockIdx.y * DG_BM, n0 = blockIdx.x * DG_BN;
  const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
  double acc[4][4] = {};
  for (int k0 = 0; k0 < g.K; k0 += DG_BK) {
    // A slab: 64 rows x 16 k -> 1024 values, 4 per thread (k fastest for coalescing)
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      int e = tid + r * 256;
      int mm = e / DG_BK, kk = e % DG_BK;
      int m = m0 + mm, k = k0 + kk;
      double v = 0.0;
      if (m < g.M && k < g.K) {
        int64_t row = g.rowidx ? int64_t(g.rowidx[m]) : int64_t(m);
        v = A[row * g.lda + k];
      }
      As[kk][mm] = v;
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      int e = tid + r * 256;
      int nn, kk;
      if (g.transB) { nn = e / DG_BK; kk = e % DG_BK; } else { kk = e / DG_BN; nn = e % DG_BN; }
      int n = n0 + nn, k = k0 + kk;
      double v = 0.0;
      if (n < g.N && k < g.K) v = g.transB ? B[int64_t(n) * g.ldb + k] : B[int64_t(k) * g.ldb + n];
      Bs[kk][nn] = v;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < DG_BK; ++kk) {
      double a[4], bb[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = As[kk][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < 4; ++j) bb[j] = Bs[kk][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fma(a[i], bb[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    int m = m0 + ty + 16 * i;
    if (m >= g.M) continue;
    int64_t row = g.rowidx ? int64_t(g.rowidx[m]) : int64_t(m);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      int n = n0 + tx + 16 * j;
      if (n >= g.N) continue;
      double* c = C + row * g.ldc + n;
      double v = g.alpha * acc[i][j];
      if (g.beta != 0.0) v = fma(g.beta, *c, v);
      *c = v;
    }
  }
}

inline cudaError_t dgemm(const DgemmArgs& g, int batch, cudaStream_t st) {
  if (g.M <= 0 || g.N <= 0 || batch <= 0) return cudaSuccess;
  dim3 grid((g.N + DG_BN - 1) / DG_BN, (g.M + DG_BM - 1) / DG_BM, batch);
  dgemm_kernel<<<grid, 256, 0, st>>>(g);
  return cudaGetLastError();
}

// The products of one A (per matrix) with every right factor of a list, C = A B + D (D null: none)
// or A B + diag I: the propagator build's FP64 products. T x T outputs per CTA, (T / 16)^2 per
// thread; the next K slab loads while one is multiplied. Bound by the FP64 pipe where the CTAs fill
// the SMs: T shrinks with the number of outputs (one CTA of 64 x 64 outputs holds an SM for 17 us a
// K slab of 16: ten products of 64 x 64 x 64 took 75 us on ten SMs).
constexpr int DG_MAXP = 4;
struct DgemmList {
  int M, K, np;
  int N[DG_MAXP], tile0[DG_MAXP + 1];  // columns, first column tile of each product
  const double* A; int64_t lda, sA;
  const double* B[DG_MAXP]; int64_t ldb[DG_MAXP], sB[DG_MAXP];
  const double* D[DG_MAXP]; int64_t ldd[DG_MAXP], sD[DG_MAXP];
  double* C[DG_MAXP]; int64_t ldc[DG_MAXP], sC[DG_MAXP];
  const double* diag[DG_MAXP];
  const int* map;  // matrix of each batch entry (null: itself)
};

template <int T>
__global__ void __launch_bounds__(256) dgemm_list_kernel(const __grid_constant__ DgemmList g) {
  constexpr int R = T / 16, L = T / 16;  // outputs per thread and side, slab values per thread and operand
  __shared__ double As[DG_BK][T + 1];
  __shared__ double Bs[DG_BK][T + 1];
  const int64_t q = g.map ? g.map[blockIdx.z] : int(blockIdx.z);
  int t = 0;
  for (int k = 1; k < g.np; ++k) t += int(blockIdx.x) >= g.tile0[k] ? 1 : 0;
  const double* A = g.A + q * g.sA;
  const double* B = g.B[t] + q * g.sB[t];
  const int m0 = blockIdx.y * T, n0 = (int(blockIdx.x) - g.tile0[t]) * T, N = g.N[t];
  const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
  double acc[R][R] = {};
  double ra[L], rb[L];
  auto load = [&](int k0) {
#pragma unroll
    for (int r = 0; r < L; ++r) {
      const int e = tid + r * 256;
      const int mm = e / DG_BK, ka = e % DG_BK, nn = e % T, kb = e / T;
      ra[r] = m0 + mm < g.M && k0 + ka < g.K ? A[int64_t(m0 + mm) * g.lda + k0 + ka] : 0.0;
      rb[r] = n0 + nn < N && k0 + kb < g.K ? B[int64_t(k0 + kb) * g.ldb[t] + n0 + nn] : 0.0;
    }
  };
  load(0);
  for (int k0 = 0; k0 < g.K; k0 += DG_BK) {
#pragma unroll
    for (int r = 0; r < L; ++r) {
      const int e = tid + r * 256;
      As[e % DG_BK][e / DG_BK] = ra[r];
      Bs[e / T][e % T] = rb[r];
    }
    __syncthreads();
    if (k0 + DG_BK < g.K) load(k0 + DG_BK);
#pragma unroll
    for (int kk = 0; kk < DG_BK; ++kk) {
      double a[R], bb[R];
#pragma unroll
      for (int i = 0; i < R; ++i) a[i] = As[kk][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < R; ++j) bb[j] = Bs[kk][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j < R; ++j) acc[i][j] = fma(a[i], bb[j], acc[i][j]);
    }
    __syncthreads();
  }
  const double* D = g.D[t] ? g.D[t] + q * g.sD[t] : nullptr;
  double* C = g.C[t] + q * g.sC[t];
#pragma unroll
  for (int i = 0; i < R; ++i) {
    const int m = m0 + ty + 16 * i;
    if (m >= g.M) continue;
#pragma unroll
    for (int j = 0; j < R; ++j) {
      const int n = n0 + tx + 16 * j;
      if (n >= N) continue;
      double v = acc[i][j];
      if (D) v += D[int64_t(m) * g.ldd[t] + n];
      else if (g.diag[t] && m == n) v += g.diag[t][q];
      C[int64_t(m) * g.ldc[t] + n] = v;
    }
  }
}

// C_t must not overlap A or any B of the call (it may be D_t).
inline cudaError_t dgemm_list(DgemmList g, int nbatch, int nsm, cudaStream_t st) {
  if (nbatch <= 0 || g.M <= 0) return cudaSuccess;
  auto tiles = [&](int T) {
    g.tile0[0] = 0;
    for (int t = 0; t < DG_MAXP; ++t) g.tile0[t + 1] = g.tile0[t] + (t < g.np ? (g.N[t] + T - 1) / T : 0);
    return dim3(unsigned(g.tile0[DG_MAXP]), unsigned((g.M + T - 1) / T), unsigned(nbatch));
  };
  auto ctas = [](dim3 d) { return int64_t(d.x) * d.y * d.z; };
  if (ctas(tiles(64)) >= 4 * nsm) dgemm_list_kernel<64><<<tiles(64), 256, 0, st>>>(g);
  else if (ctas(tiles(32)) >= 2 * nsm) dgemm_list_kernel<32><<<tiles(32), 256, 0, st>>>(g);
  else dgemm_list_kernel<16><<<tiles(16), 256, 0, st>>>(g);
  return cudaGetLastError();
}

}  // namespace lem
