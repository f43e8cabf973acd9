// Dense FP64 matrix products of the propagator build on the tcgen05 tensor cores (Sec. 1, Sec. 4:
// Pade-13 products, the denominator solve's trailing updates and the squarings of scaling and
// squaring), for the split-precision tiers, as sums of digit products (oz_core.cuh, coarse
// digits). The FP64 tier keeps FP64 multiply-adds: its propagators hold the entries of FP64 range
// far from the owner, which digits below the largest of a row do not.
//
// One call multiplies one A (per class) by up to four B: the Pade evaluation and the squarings
// multiply several matrices by the same left factor, which is then cut once and whose products
// fill the SMs together. Two launches a call: digits of A and of every B, then the products.
//
// The dropped digits and sums are below 2^-48 of sum_k |A_ik| |B_kj| at the operands' scale. A row
// of A or column of B that holds an infinity or a NaN gives NaN.
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <new>
#include <string>

#include "lem_internal.h"
#include "oz_core.cuh"

namespace lem {

namespace {

constexpr int MAXP = 4;             // right factors per call
constexpr int CUT_THREADS = 256;

// Strided batch of row-major FP64 matrices: element (q, r, c) at p + map(q) stride + r ld + c.
struct Mat {
  const double* p;
  int64_t ld, stride;
};

// Matrix q of a product batch is matrix map[q] of the caller's arrays (map null: q itself);
// digits and exponents are stored at q.
__device__ __forceinline__ int mat_of(const int* map, int q) { return map ? map[q] : q; }

__device__ __forceinline__ unsigned long long bits_of(double x) {
  return static_cast<unsigned long long>(__double_as_longlong(x));
}

struct CutParams {
  Mat A, B[MAXP];
  int rows, kdim;          // A rows x kdim
  int cols[MAXP];          // each B kdim x cols
  int tile0[MAXP + 1];     // its first tile of 64 columns; the last entry: tiles in all
  int m_pad, nkb;
  const int* map;
  int* e;                  // [batch][m_pad]
  int* f;                  // [batch][tiles][64]
  __half* sa;              // [batch][m_pad / 128][nkb] blocks
  __half* sb;              // [batch][tiles][nkb] blocks
};

// The product that column tile t belongs to.
template <class P>
__device__ __forceinline__ int product_of(const P& p, int t) {
  int b = 0;
#pragma unroll
  for (int k = 1; k < MAXP; ++k) b += t >= p.tile0[k] ? 1 : 0;
  return b;
}

// Digits of A (a CTA per 8 rows) and of the B's (a CTA per 64 columns, which it reads twice: the
// largest exponents, then the digits). blockIdx.x: row groups of A, then column blocks of the
// B's. Bound by the 14 bytes written per element.
__global__ void __launch_bounds__(CUT_THREADS) oz_cut_kernel(const __grid_constant__ CutParams p) {
  const int q = blockIdx.y, tid = threadIdx.x;
  const int64_t src = mat_of(p.map, q);
  const int row_groups = p.m_pad / 8;
  if (int(blockIdx.x) < row_groups) {
    const int r0 = int(blockIdx.x) * 8, warp = tid / 32, lane = tid % 32;
    __shared__ int ex[8];
    {
      const int i = r0 + warp;
      int E = 0;
      if (i < p.rows) {
        const double* row = p.A.p + src * p.A.stride + int64_t(i) * p.A.ld;
#pragma unroll 4
        for (int k = lane; k < p.kdim; k += 32) E = max(E, oz::exp_field(bits_of(row[k])));
      }
      for (int o = 16; o > 0; o >>= 1) E = max(E, __shfl_xor_sync(0xffffffffu, E, o));
      if (lane == 0) {
        ex[warp] = oz::scale_exp(E);
        p.e[size_t(q) * p.m_pad + i] = ex[warp];
      }
    }
    __syncthreads();
    // 32 lanes: 4 rows x 8 K chunks, so a warp reads runs of 512 bytes
    const int r = (tid / 8) % 8, i = r0 + r;
    const bool live = i < p.rows;
    const int er = ex[r] == oz::kNonFinite ? 4096 : ex[r];
    const double* row = p.A.p + src * p.A.stride + int64_t(live ? i : 0) * p.A.ld;
    __half* dst = p.sa + (size_t(q) * (p.m_pad / oz::BM) + i / oz::BM) * size_t(p.nkb) * oz::A_BLOCK;
    for (int k8 = ((tid / 64) * 8 + tid % 8) * 8; k8 < p.nkb * oz::KB; k8 += CUT_THREADS) {
      int N[8][oz::S];
#pragma unroll
      for (int u = 0; u < 8; ++u) oz::coarse_digits(live && k8 + u < p.kdim ? bits_of(row[k8 + u]) : 0ull, er, N[u]);
      oz::store_coarse_digits(dst + size_t(k8 / oz::KB) * oz::A_BLOCK + oz::tile_off(i % oz::BM, k8 % oz::KB), oz::A_SLICE, N);
    }
    return;
  }
  const int ct = int(blockIdx.x) - row_groups, b = product_of(p, ct), tiles = p.tile0[MAXP];
  const int c = tid % oz::BN, j = (ct - p.tile0[b]) * oz::BN + c, g = tid / oz::BN;  // 4 groups of 64 columns
  const bool live = j < p.cols[b];
  const double* col = p.B[b].p + src * p.B[b].stride + (live ? j : 0);
  const int64_t ld = p.B[b].ld;
  __shared__ int fx[oz::BN];
  if (tid < oz::BN) fx[tid] = 0;
  __syncthreads();
  int E = 0;
  if (live) {
#pragma unroll 8
    for (int k = g; k < p.kdim; k += CUT_THREADS / oz::BN) E = max(E, oz::exp_field(bits_of(col[int64_t(k) * ld])));
    atomicMax(&fx[c], E);
  }
  __syncthreads();
  const int sc = oz::scale_exp(fx[c]);
  if (g == 0) p.f[(size_t(q) * tiles + ct) * oz::BN + c] = sc;
  const int ec = sc == oz::kNonFinite ? 4096 : sc;
  __half* dst = p.sb + (size_t(q) * tiles + ct) * size_t(p.nkb) * oz::B_BLOCK;
  for (int k8 = g * 8; k8 < p.nkb * oz::KB; k8 += CUT_THREADS / oz::BN * 8) {
    int N[8][oz::S];
#pragma unroll
    for (int u = 0; u < 8; ++u)
      oz::coarse_digits(live && k8 + u < p.kdim ? bits_of(col[int64_t(k8 + u) * ld]) : 0ull, ec, N[u]);
    oz::store_coarse_digits(dst + size_t(k8 / oz::KB) * oz::B_BLOCK + oz::tile_off(c, k8 % oz::KB), oz::B_SLICE, N);
  }
}

struct MulParams {
  int M, m_pad, nkb;
  int cols[MAXP], tile0[MAXP + 1];
  const __half* sa;
  const __half* sb;
  const int* map;
  const int* e;
  const int* f;
  Mat D[MAXP];             // addends (may alias C; p null: none)
  double* C[MAXP];
  int64_t ldc[MAXP], sC[MAXP];
  const double* diag[MAXP];  // per matrix: added to the diagonal of C (null: none)
  int zr0, zr1;            // rows [zr0, zr1) of D read as zero
  int* err;
};

// The units of one CTA of the product kernel: 128 x 64 output tiles, every gridDim.x-th. Tiles of
// one row block are consecutive, so CTAs that run together share A's digits in L2.
struct MulWork {
  const MulParams& p;
  int units, mt, tiles;
  int (*s_e)[oz::BM];  // [2] scale exponents of the tile's rows and columns, by the unit's parity
  int (*s_f)[oz::BN];
  struct Unit { int q, mb, ct; };  // matrix, row block, column tile
  __device__ Unit unit(int k) const {
    int t = int(blockIdx.x) + k * int(gridDim.x);
    Unit u;
    u.ct = t % tiles;
    t /= tiles;
    u.mb = t % mt;
    u.q = t / mt;
    return u;
  }
  __device__ int count() const { return (units - int(blockIdx.x) + int(gridDim.x) - 1) / int(gridDim.x); }
  __device__ oz::Tile tile(int k) const {
    const Unit u = unit(k);
    return {p.sa + (size_t(u.q) * mt + u.mb) * size_t(p.nkb) * oz::A_BLOCK,
            p.sb + (size_t(u.q) * tiles + u.ct) * size_t(p.nkb) * oz::B_BLOCK, p.nkb};
  }
  __device__ void begin(int k) const {
    const Unit u = unit(k);
    const int t = int(threadIdx.x) - 64;
    if (t < oz::BM) s_e[k & 1][t] = p.e[size_t(u.q) * p.m_pad + u.mb * oz::BM + t];
    else if (t < oz::BM + oz::BN)
      s_f[k & 1][t - oz::BM] = p.f[(size_t(u.q) * tiles + u.ct) * oz::BN + t - oz::BM];
    oz::epi_sync();
  }
  // C = sums + D + diag, element by element (D and C have one leading dimension)
  struct Out {
    const int* e;
    const int* f;
    const double* D;
    double* C;
    int64_t ld;
    const double* dg;  // (without D)
    int i0, j0, M, N, zr0, zr1;
    __device__ int scale(int row, int col) const { return e[row] + f[col] - 14; }
    __device__ double value(int row, int col, double v) const {
      return e[row] == oz::kNonFinite || f[col] == oz::kNonFinite ? __longlong_as_double(0x7FF8000000000000ll) : v;
    }
    __device__ int64_t row_at(int row) const { return i0 + row < M ? int64_t(i0 + row) * ld : -1; }
    __device__ int64_t col_at(int col) const { return j0 + col < N ? j0 + col : INT64_MIN / 2; }
    __device__ double load(int64_t at, int row) const {
      if (D) return i0 + row < zr0 || i0 + row >= zr1 ? D[at] : 0.0;
      return dg && at == int64_t(i0 + row) * (ld + 1) ? *dg : 0.0;
    }
    __device__ void store(int64_t at, double y, double old) const {
      C[at] = D || dg != nullptr ? y + old : y;
    }
  };
  __device__ void finish(int k, int quarter, int half, int lane, double* out, const float (&hi)[32],
                         const float (&lo)[32]) const {
    const Unit u = unit(k);
    const int64_t m = mat_of(p.map, u.q);
    const int b = product_of(p, u.ct), i0 = u.mb * oz::BM, j0 = (u.ct - p.tile0[b]) * oz::BN;
    const Out o{s_e[k & 1], s_f[k & 1], p.D[b].p ? p.D[b].p + m * p.D[b].stride : nullptr, p.C[b] + m * p.sC[b],
                p.ldc[b], p.diag[b] && i0 < j0 + oz::BN && j0 < i0 + oz::BM ? p.diag[b] + m : nullptr, i0, j0, p.M,
                p.cols[b], p.zr0, p.zr1};
    oz::write_tile(o, quarter, half, lane, out, hi, lo);
  }
};

__global__ void __launch_bounds__(oz::THREADS, 1) oz_mul_kernel(const __grid_constant__ MulParams p, int units) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  __shared__ volatile int s_abort;
  __shared__ int s_e[2][oz::BM], s_f[2][oz::BN];
  const oz::Shared sh = oz::carve(smem_raw);
  const uint32_t tmem = oz::setup(sh, &s_abort);
  MulWork work{p, units, p.m_pad / oz::BM, p.tile0[MAXP], s_e, s_f};
  oz::run<oz::Coarse>(sh, tmem, work, p.err, &s_abort);
  oz::release(tmem);
}

inline int pad_to(int x, int m) { return (x + m - 1) / m * m; }

struct Caps {
  size_t a, b, e, f;
};
// Room for products of np right factors of n x n, and for the rank-64 updates of an n x gjcols
// elimination (of rank n where n is less).
Caps caps_for(int n, int nb, int gjcols, int np) {
  const size_t ka = pad_to(n, oz::KB) / oz::KB, ra = pad_to(n, oz::BM) / oz::BM, cb = pad_to(n, oz::BN) / oz::BN,
               cg = pad_to(std::max(gjcols, 1), oz::BN) / oz::BN;
  return {size_t(nb) * ra * ka * oz::A_BLOCK, size_t(nb) * std::max(np * cb * ka, cg * std::min<size_t>(ka, 64 / oz::KB)) * oz::B_BLOCK,
          size_t(nb) * ra * oz::BM, size_t(nb) * std::max(np * cb, cg) * oz::BN};
}

}  // namespace

// Workspace of one build batch: digits of A and of the B's, exponents.
struct TcGemm {
  int nb = 0;
  int nsm = 152;
  Caps cap{};
  __half* sa = nullptr;
  __half* sb = nullptr;
  int* e = nullptr;
  int* f = nullptr;
  int* err = nullptr;
};

size_t tc_gemm_bytes(int n, int nb, int gjcols, int np) {
  const Caps c = caps_for(n, nb, gjcols, np);
  return sizeof(__half) * (c.a + c.b) + sizeof(int) * (c.e + c.f) + 256;
}

void tc_gemm_destroy(TcGemm* g) { delete g; }

// mem: tc_gemm_bytes of device memory (256-byte aligned) that outlives the workspace
lem_status tc_gemm_create(int n, int nb, int gjcols, int np, void* mem, cudaStream_t st, TcGemm** out) {
  *out = nullptr;
  // the shared-memory attribute is per device (cheap to set again)
  if (cudaFuncSetAttribute(oz_mul_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, oz::SMEM) != cudaSuccess)
    return cuda_fail(cudaGetLastError(), "oz_mul_kernel attributes");
  TcGemm* g = new (std::nothrow) TcGemm();
  if (!g) return fail(LEM_ENOMEM, "host allocation failed");
  const Caps c = caps_for(n, nb, gjcols, np);
  g->nb = nb;
  g->cap = c;
  int dev = 0, nsm = 0;
  if (cudaGetDevice(&dev) == cudaSuccess &&
      cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && nsm > 0)
    g->nsm = nsm;
  // (every part but the last is a whole number of digit blocks or of 64 integers)
  g->sa = static_cast<__half*>(mem);
  g->sb = g->sa + c.a;
  g->e = reinterpret_cast<int*>(g->sb + c.b);
  g->f = g->e + c.e;
  g->err = g->f + c.f;
  if (cudaMemsetAsync(g->err, 0, sizeof(int), st) != cudaSuccess) {
    tc_gemm_destroy(g);
    return cuda_fail(cudaGetLastError(), "tensor-core build workspace");
  }
  *out = g;
  return LEM_OK;
}

// C_t[m] = A[m] B_t[m] + D_t[m] (+ diag_t[m] I) for every product t of the list and m = map[q],
// q < nbatch (map a device array, or null for m = q): A is M x K, B_t K x N, C_t and D_t M x N,
// row-major FP64 with the given leading dimensions and batch strides; D null: no addend, D rows
// [zr0, zr1) taken as zero. All operands are cut before the products run, so a C may overlap
// them; D_t may alias C_t.
lem_status tc_gemm(TcGemm* g, int nbatch, const int* map, int M, int K, const double* A, int64_t lda, int64_t sA,
                   const TcProduct* list, int np, int zr0, int zr1, cudaStream_t st) {
  if (nbatch <= 0 || M <= 0) return LEM_OK;
  const int m_pad = pad_to(M, oz::BM), nkb = pad_to(std::max(K, 1), oz::KB) / oz::KB;
  int tiles = 0;
  for (int t = 0; t < std::min(np, MAXP); ++t) tiles += pad_to(list[t].N, oz::BN) / oz::BN;
  if (tiles == 0) return LEM_OK;
  if (np < 1 || np > MAXP || nbatch > g->nb || size_t(nbatch) * (m_pad / oz::BM) * nkb * oz::A_BLOCK > g->cap.a ||
      size_t(nbatch) * tiles * nkb * oz::B_BLOCK > g->cap.b || size_t(nbatch) * m_pad > g->cap.e ||
      size_t(nbatch) * tiles * oz::BN > g->cap.f)
    return fail(LEM_EINVAL, "tensor-core product larger than its workspace");
  CutParams c{};
  MulParams m{};
  c.A = Mat{A, lda, sA};
  c.rows = m.M = M;
  c.kdim = K;
  c.m_pad = m.m_pad = m_pad;
  c.nkb = m.nkb = nkb;
  c.map = m.map = map;
  c.e = g->e;
  c.f = g->f;
  c.sa = g->sa;
  c.sb = g->sb;
  m.e = g->e;
  m.f = g->f;
  m.sa = g->sa;
  m.sb = g->sb;
  m.zr0 = zr0;
  m.zr1 = zr1;
  m.err = g->err;
  for (int t = 0; t < np; ++t) {
    const TcProduct& q = list[t];
    if (q.D && (q.ldd != q.ldc || q.diag))
      return fail(LEM_EINVAL, "an addend has the result's leading dimension and no diagonal term beside it");
    c.cols[t] = m.cols[t] = q.N;
    c.tile0[t + 1] = m.tile0[t + 1] = c.tile0[t] + pad_to(q.N, oz::BN) / oz::BN;
    c.B[t] = Mat{q.B, q.ldb, q.sB};
    m.D[t] = Mat{q.D, q.ldd, q.sD};
    m.C[t] = q.C;
    m.ldc[t] = q.ldc;
    m.sC[t] = q.sC;
    m.diag[t] = q.diag;
  }
  for (int t = np; t < MAXP; ++t) c.tile0[t + 1] = m.tile0[t + 1] = tiles;  // (none)
  oz_cut_kernel<<<dim3(unsigned(m_pad / 8 + tiles), unsigned(nbatch)), CUT_THREADS, 0, st>>>(c);
  LEM_CUDA_TRY(cudaGetLastError());
  const int units = nbatch * (m_pad / oz::BM) * tiles;
  oz_mul_kernel<<<std::min(units, g->nsm), oz::THREADS, oz::SMEM, st>>>(m, units);
  LEM_CUDA_TRY(cudaGetLastError());
  return LEM_OK;
}

// Error flag of the workspace's products (reads it after synchronising st).
lem_status tc_gemm_check(TcGemm* g, cudaStream_t st) {
  int e = 0;
  LEM_CUDA_TRY(cudaMemcpyAsync(&e, g->err, sizeof(int), cudaMemcpyDeviceToHost, st));
  LEM_CUDA_TRY(cudaStreamSynchronize(st));
  if (e != 0) {
    cudaMemsetAsync(g->err, 0, sizeof(int), st);
    return fail(LEM_ETIMEOUT, "tensor-core build product gave up waiting on an mbarrier (code " +
                                  std::to_string(e) + ")");
  }
  return LEM_OK;
}

}  // namespace lem
