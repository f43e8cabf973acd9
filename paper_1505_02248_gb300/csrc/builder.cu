// Local propagator builder (Sec. 3 step 2; Pade approximation with scaling and squaring
// as named in Sec. 1 and Sec. 4), batched over propagator classes, in FP64. The matrix
// products of the split-precision tiers run on the tensor cores as sums of digit products
// (builder_tc.cu, about 2^-45 relative to the operands' scale), those of the FP64 tier on the FP64
// pipe; the pivots of the Pade denominator solve are FP64 either way.
//
// For each class the local matrix X = dt A_M (principal submatrix on the window, i.e.
// Dirichlet data at the artificial boundary; plus dt diag(1 - 3u^2) with the reaction, or
// times diag(phi'(u)) on the right for the porous-medium equation) is
// assembled in a zero-padded n x n frame (padding is an exact block-diagonal embedding).
//   EXP:  P = R_D exp(X)
//   PHI:  P = R_D phi_1(X), the top-right block of exp(Z), Z = [[X, I], [0, 0]].
// The PHI path never forms the 2n x 2n matrix Z: every power and polynomial of Z has the
// form (T, B; beta) = [[T, B], [0, beta I]], and products of such pairs need two n x n
// products. Degree-13 Pade (Higham 2005 coefficients b_j = (2m-j)! m! / ((2m)! j! (m-j)!)),
// s = smallest integer >= 0 with ||Z||_1 / 2^s <= theta_13 from the exact 1-norm,
// (V - U) R = (V + U) by Gauss-Jordan elimination with partial pivoting, then s squarings.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdlib>
#include <numeric>
#include <string>
#include <vector>

#include <cooperative_groups.h>
#include <nvtx3/nvToolsExt.h>

#include "dgemm.cuh"
#include "lem_internal.h"

namespace lem {

namespace {

constexpr double kTheta13 = 5.371920351148152;

// b_j for m = 13 as exact rationals (numerator integers / 64764752532480000).
const double kPadeInt[14] = {64764752532480000.0, 32382376266240000.0, 7771770303897600.0,
                             1187353796428800.0,  129060195264000.0,   10559470521600.0,
                             670442572800.0,      33522128640.0,       1323241920.0,
                             40840800.0,          960960.0,            16380.0,
                             182.0,               1.0};

struct BatchClass {
  TileDesc rep;      // representative tile (window geometry)
  int32_t whole[2];
};

// ---------------------------------------------------------------- assembly
// X is zero on entry. nonlin 1: + dt diag(1 - 3u^2); nonlin 2 (porous medium): X diag(phi'(u)) with
// phi'(u) = m |u|^(m-1), each entry scaled by phi' at its column's node.
__global__ void assemble_local_kernel(double* X, int n, const BatchClass* bc, int nb,
                                      const double* coef, int64_t cstride, int64_t ny,
                                      int64_t nx, int ndim, const double* u, double dt,
                                      int nonlin, double pm) {
  const int b = blockIdx.y;
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= nb || k >= n) return;
  double* row = X + (int64_t(b) * n + k) * n;
  const BatchClass c = bc[b];
  const int wy = c.rep.wext[0], wx = c.rep.wext[1];
  if (k >= wy * wx) return;  // padding row
  const int a = k / wx, bb = k % wx;
  int64_t gy = (int64_t(c.rep.org[0]) + a) % ny;
  if (gy < 0) gy += ny;
  int64_t gx = (int64_t(c.rep.org[1]) + bb) % nx;
  if (gx < 0) gx += nx;
  const int64_t p = gy * nx + gx;
  const int64_t npts = ny * nx;
  auto cf = [&](int which) { return coef[which * (cstride ? npts : 1) + (cstride ? p : 0)]; };
  const bool porous = u && nonlin == 2;
  // phi'(u) at global node q (1 unless porous)
  auto dphi = [&](int64_t q) { return porous ? pm * abs_pow(u[q], pm - 1.0) : 1.0; };
  // the four neighbours' global nodes (wrapped; a window never holds a node beyond a wall)
  const int64_t qw = gy * nx + (gx + nx - 1) % nx, qe = gy * nx + (gx + 1) % nx;
  const int64_t qs = ((gy + ny - 1) % ny) * nx + gx, qn = ((gy + 1) % ny) * nx + gx;
  double diag = cf(0);
  if (u && nonlin == 1) diag += dt * (1.0 - 3.0 * u[p] * u[p]);
  row[k] += diag * dphi(p);
  // W (x - 1) and E (x + 1): inside the window, or wrapped when it spans the periodic axis
  if (bb >= 1) row[k - 1] += cf(1) * dphi(qw);
  else if (c.whole[1]) row[k + wx - 1] += cf(1) * dphi(qw);
  if (bb + 1 < wx) row[k + 1] += cf(2) * dphi(qe);
  else if (c.whole[1]) row[k + 1 - wx] += cf(2) * dphi(qe);
  if (ndim == 2) {
    if (a >= 1) row[k - wx] += cf(3) * dphi(qs);
    else if (c.whole[0]) row[k + (wy - 1) * wx] += cf(3) * dphi(qs);
    if (a + 1 < wy) row[k + wx] += cf(4) * dphi(qn);
    else if (c.whole[0]) row[k - (wy - 1) * wx] += cf(4) * dphi(qn);
  }
}

// Complex problems: the real embedding [[Re X, -Im X], [Im X, Re X]] of X = dt A_M (n = twice
// the window nodes): row k carries the real part of node k's equation, row n/2 + k the
// imaginary part. Coefficients: real parts at coef[w], imaginary parts at coef[5 + w].
__global__ void assemble_local_complex_kernel(double* X, int n, const BatchClass* bc, int nb, const double* coef,
                                              int64_t cstride, int64_t ny, int64_t nx, int ndim) {
  const int b = blockIdx.y;
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  const int h = n / 2;
  if (b >= nb || k >= h) return;
  double* rr = X + (int64_t(b) * n + k) * n;
  double* ri = X + (int64_t(b) * n + h + k) * n;
  const BatchClass c = bc[b];
  const int wy = c.rep.wext[0], wx = c.rep.wext[1];
  if (k >= wy * wx) return;  // padding node
  const int a = k / wx, bb = k % wx;
  int64_t gy = (int64_t(c.rep.org[0]) + a) % ny;
  if (gy < 0) gy += ny;
  int64_t gx = (int64_t(c.rep.org[1]) + bb) % nx;
  if (gx < 0) gx += nx;
  const int64_t p = gy * nx + gx, npts = ny * nx;
  auto add = [&](int col, int w) {
    const int64_t o = cstride ? p : 0;
    const double cr = coef[int64_t(w) * (cstride ? npts : 1) + o];
    const double ci = coef[int64_t(5 + w) * (cstride ? npts : 1) + o];
    rr[col] += cr;
    rr[h + col] -= ci;
    ri[col] += ci;
    ri[h + col] += cr;
  };
  add(k, 0);
  if (bb >= 1) add(k - 1, 1);
  else if (c.whole[1]) add(k + wx - 1, 1);
  if (bb + 1 < wx) add(k + 1, 2);
  else if (c.whole[1]) add(k + 1 - wx, 2);
  if (ndim == 2) {
    if (a >= 1) add(k - wx, 3);
    else if (c.whole[0]) add(k + (wy - 1) * wx, 3);
    if (a + 1 < wy) add(k + wx, 4);
    else if (c.whole[0]) add(k - (wy - 1) * wx, 4);
  }
}

// column 1-norms -> per-matrix max (non-negative doubles order like their bit patterns); a block
// takes 32 columns, 8 threads a column
__global__ void __launch_bounds__(256) norm1_kernel(const double* X, int n, unsigned long long* out) {
  const int b = blockIdx.y;
  const int c = threadIdx.x % 32, g = threadIdx.x / 32, j = blockIdx.x * 32 + c;
  __shared__ double part[8][32];
  const double* M = X + int64_t(b) * n * n;
  double s = 0.0;
  if (j < n) {
#pragma unroll 8
    for (int i = g; i < n; i += 8) s += fabs(M[int64_t(i) * n + j]);
  }
  part[g][c] = s;
  __syncthreads();
  if (g == 0 && j < n) {
    for (int q = 1; q < 8; ++q) s += part[q][c];
    atomicMax(out + b, (unsigned long long)__double_as_longlong(s));
  }
}

// X <- X c and B2 <- X c^2 (c = 2^-s per matrix; B2 null: not wanted)
__global__ void scale_kernel(double* X, double* B2, int64_t nn, const double* c) {
  const int b = blockIdx.y;
  const int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (e >= nn) return;
  const double v = X[b * nn + e] * c[b];
  X[b * nn + e] = v;
  if (B2) B2[b * nn + e] = v * c[b];
}

// The linear combinations of the Pade-13 evaluation in one pass over the powers:
//   W = b13 Z6 + b11 Z4 + b9 Z2,  A3 = b7 Z6 + b5 Z4 + b3 Z2 (+ b1 I),
//   V = b12 Z6 + b10 Z4 + b8 Z2,  VT = b6 Z6 + b4 Z4 + b2 Z2 (+ b0 I);
// blockIdx.z 0: the T blocks (diagonal terms), 1: the B blocks (V's is not needed: it cancels in
// the solve's right-hand side). Bound by the FP64 pipe (12
// multiply-adds per element); one pass per combination read the powers four times over.
struct PadeTerms {
  const double* z2[2];
  const double* z4[2];
  const double* z6[2];
  double* w[2];
  double* a3[2];
  double* v[1];
  double* vt[1];
  double b[14];
};
__global__ void pade_terms_kernel(const __grid_constant__ PadeTerms p, int n, int64_t total) {
  const int h = blockIdx.z;
  const int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (e >= total) return;
  const double z2 = p.z2[h][e], z4 = p.z4[h][e], z6 = p.z6[h][e];
  const int64_t nn = int64_t(n) * n;
  const unsigned in = unsigned(e % nn);
  const bool dg = h == 0 && in / unsigned(n) == in % unsigned(n);
  p.w[h][e] = fma(p.b[9], z2, fma(p.b[11], z4, p.b[13] * z6));
  double a = fma(p.b[3], z2, fma(p.b[5], z4, p.b[7] * z6));
  if (dg) a += p.b[1];
  p.a3[h][e] = a;
  if (h) return;
  p.v[0][e] = fma(p.b[8], z2, fma(p.b[10], z4, p.b[12] * z6));
  double t = fma(p.b[2], z2, fma(p.b[4], z4, p.b[6] * z6));
  if (dg) t += p.b[0];
  p.vt[0][e] = t;
}

// G = [V_T - U_T | V_T + U_T | 2 U_B] (UB null: no third block)
__global__ void solve_system_kernel(double* G, int n, int gjcols, const double* VT, const double* UT,
                                    const double* UB) {
  const int b = blockIdx.y;
  const int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x, nn = int64_t(n) * n;
  if (e >= nn) return;
  const int i = int(e / n), j = int(e % n);
  const double v = VT[b * nn + e], u = UT[b * nn + e];
  double* row = G + (int64_t(b) * n + i) * gjcols + j;
  row[0] = v - u;
  row[n] = v + u;
  if (UB) row[2 * n] = 2.0 * UB[b * nn + e];
}

// out[b] = sum_t w_t in_t[b] + diag * dscale[b] * I   (dscale may be null: 1)
struct Lin {
  const double* in[4];
  double w[4];
  int nin;
  double diag;
  const double* dscale;
  const double* wscale0;  // optional per-batch multiplier of w[0]
};

__global__ void lincomb_kernel(double* out, int n, int64_t ld, int ncols, Lin L) {
  const int b = blockIdx.y;
  const int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (e >= int64_t(n) * ncols) return;
  const int i = int(e / ncols), j = int(e % ncols);
  const int64_t off = int64_t(b) * n * ld + int64_t(i) * ld + j;
  double v = 0.0;
  for (int t = 0; t < L.nin; ++t) {
    double w = L.w[t];
    if (t == 0 && L.wscale0) w *= L.wscale0[b];
    v += w * L.in[t][off];
  }
  if (i == j && L.diag != 0.0) v += L.diag * (L.dscale ? L.dscale[b] : 1.0);
  out[off] = v;
}

// ---------------------------------------------------------------- blocked Gauss-Jordan
// Gauss-Jordan elimination with partial pivoting on G = [Q | RHS] (n x gjcols, row-major), in panels
// of GJ_KB columns. The panel's GJ_KB pivot steps (partial pivoting, FP64) are applied to the panel columns and to a tracker
// Y (n x GJ_KB): at step c, right after the row swap, Y[k0 + c][c] = 1 is injected, and every
// later swap, scaling and elimination acts on Y too. At the end of the panel the composite row
// operation is M = T Pi with T = I + W E_K^T (Pi: the panel's swaps, K: rows k0 .. k0 + kb),
// and Y = T[:, K], so any other column becomes
//   rows K:      Y_K (Pi G)[K, :]
//   other rows:  (Pi G)[i, :] + Y_i (Pi G)[K, :],
// one rank-kb product C = Y B + D with B the permuted pivot rows and D the permuted columns with
// rows K taken as zero, on the tensor cores or (FP64 tier) as an FP64 product; one pivot at a time
// every pivot read and wrote all of G. (One product of rank 256 for four panels saves a tenth of a build
// of 25 matrices of 784, but rounds worse: 1.5 to 2.6 times the error of the propagators.)
constexpr int GJ_KB = 64;

// One pivot step of a panel at columns k0 .. of the matrix, copied to Y (n x GJ_KB), for matrices too large for
// bgj_panel_kernel. In place: the pivot column becomes the tracker column.
__global__ void bgj_pivot_kernel(double* Y, int n, int k0, int c, int kb, int* piv, int* status) {
  const int b = blockIdx.x;
  double* M = Y + int64_t(b) * n * GJ_KB;
  const int r = k0 + c;
  __shared__ double sv[256];
  __shared__ int si[256];
  double best = -1.0;
  int bi = r;
  for (int i = r + threadIdx.x; i < n; i += blockDim.x) {
    const double v = fabs(M[int64_t(i) * GJ_KB + c]);
    if (v > best) { best = v; bi = i; }
  }
  sv[threadIdx.x] = best;
  si[threadIdx.x] = bi;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) {
      const double o = sv[threadIdx.x + s];
      const int oi = si[threadIdx.x + s];
      if (o > sv[threadIdx.x] || (o == sv[threadIdx.x] && oi < si[threadIdx.x])) {
        sv[threadIdx.x] = o;
        si[threadIdx.x] = oi;
      }
    }
    __syncthreads();
  }
  const int p = si[0];
  const double pv = M[int64_t(p) * GJ_KB + c];
  __syncthreads();  // every thread holds pv before rows r / p are rewritten
  if (!(sv[0] > 0.0) || !isfinite(pv)) {
    if (threadIdx.x == 0) {
      atomicExch(status, int(LEM_ENUMERIC));
      piv[b * GJ_KB + c] = r;  // no swap
    }
    return;
  }
  if (threadIdx.x == 0) piv[b * GJ_KB + c] = p;
  const double inv = 1.0 / pv;
  for (int j = threadIdx.x; j < kb; j += blockDim.x) {
    const double a = M[int64_t(r) * GJ_KB + j], q = M[int64_t(p) * GJ_KB + j];
    if (p != r) M[int64_t(p) * GJ_KB + j] = a;
    M[int64_t(r) * GJ_KB + j] = (j == c ? 1.0 : q) * inv;  // inject the unit column, then scale
  }
}

// Eliminate panel column c from every row but the pivot row: 4 rows per block, thread t of a row
// updates panel column t.
__global__ void bgj_elim_kernel(double* Y, int n, int k0, int c, int kb) {
  const int b = blockIdx.y;
  const int i = blockIdx.x * 4 + threadIdx.x / 64, t = threadIdx.x % 64;
  const int r = k0 + c;
  double* M = Y + int64_t(b) * n * GJ_KB;
  const bool live = i < n && i != r;
  const double f = live ? M[int64_t(i) * GJ_KB + c] : 0.0;
  __syncthreads();  // column c is read before it is overwritten
  if (!live || f == 0.0 || t >= kb) return;
  double* m = M + int64_t(i) * GJ_KB + t;
  *m = fma(-f, M[int64_t(r) * GJ_KB + t], t == c ? 0.0 : *m);
}

// A whole panel in one launch, a cluster of CTAs per matrix, each holding a share of the panel's
// rows in shared memory. The panel's columns are overwritten by the tracker as they are
// eliminated (a pivot column is no longer needed once its tracker column begins), so each pivot
// step is one update of the share: M[i][j] -= M[i][c] M[r][j], with column c taken as zero before
// it. Per step every CTA writes its best pivot candidate with that candidate's row (and the holder
// of row r that row) into every other's shared memory, one cluster barrier follows, and every CTA
// picks the same winner from its own copy. Bound by the chain of a step (reduction, barrier,
// reciprocal) and by the FP64 pipe for the update, 2 multiply-adds per clock and SM. Two launches
// per pivot column (kept for matrices beyond PANEL_MAX_N) cost 17 us on 25 matrices of 784 nodes.
// Updating the next pivot's column first, to search it during the update, gained nothing.
constexpr int PANEL_THREADS = 256, PANEL_PITCH = GJ_KB + 1, PANEL_MAX_CLUSTER = 8, PANEL_MAX_ROWS = 360;
constexpr int PANEL_MAX_N = PANEL_MAX_CLUSTER * PANEL_MAX_ROWS;

struct PanelPub {
  double cand[GJ_KB];  // the candidate's row
  long long val;       // its magnitude (the bits)
  int idx;
  int pad;
};
struct PanelStep {
  PanelPub from[PANEL_MAX_CLUSTER];
  double rrow[GJ_KB];  // row r
};

// src: the panel's columns (leading dimension lds, matrices ss apart); Y: where the tracker goes.
__global__ void __launch_bounds__(PANEL_THREADS) bgj_panel_kernel(const double* src, int64_t lds, int64_t ss, int n,
                                                                  int k0, int kb, int csize, int rows_per, double* Y,
                                                                  int* piv, int* status) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  extern __shared__ __align__(16) double psm[];
  PanelStep* steps = reinterpret_cast<PanelStep*>(psm);  // [2], by the step's parity
  double* prow = psm + 2 * sizeof(PanelStep) / sizeof(double);  // [GJ_KB] the scaled pivot row
  double* M = prow + GJ_KB;                           // [rows_per][PANEL_PITCH]
  double* fcol = M + size_t(rows_per) * PANEL_PITCH;  // [rows_per] column c before the step
  int* fzero = reinterpret_cast<int*>(fcol + rows_per);  // [rows_per] whether it is zero there (kept as it is:
                                                         // an FP64 comparison costs as much as the update)
  __shared__ long long wv[PANEL_THREADS / 32];
  __shared__ int wi[PANEL_THREADS / 32];
  const int b = blockIdx.x / csize, rank = blockIdx.x % csize;
  const int lo = rank * rows_per, cnt = max(0, min(rows_per, n - lo));
  const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
  const double* Sb = src + int64_t(b) * ss;
  for (int e = tid; e < cnt * GJ_KB; e += PANEL_THREADS) {
    const int i = e / GJ_KB, j = e % GJ_KB;
    if (j < kb) M[i * PANEL_PITCH + j] = Sb[int64_t(lo + i) * lds + j];
  }
  cl.sync();  // every CTA of the cluster runs before its memory is written
  const int j = tid % GJ_KB, grp = tid / GJ_KB;
  for (int c = 0; c < kb; ++c) {
    const int r = k0 + c;
    PanelStep& st = steps[c & 1];
    // this CTA's largest |M[i][c]|, i >= r (the smallest row of equals); magnitudes compare as
    // integers, a NaN never wins
    long long best = -1;
    int bi = n;
    for (int i = tid; i < cnt; i += PANEL_THREADS) {
      const double v = M[i * PANEL_PITCH + c];
      fcol[i] = v;
      const long long m = __double_as_longlong(v) & 0x7FFFFFFFFFFFFFFFll;
      fzero[i] = m == 0;
      if (lo + i >= r && m > best && m <= 0x7FF0000000000000ll) {
        best = m;
        bi = lo + i;
      }
    }
    for (int o = 16; o > 0; o >>= 1) {
      const long long ov = __shfl_xor_sync(0xffffffffu, best, o);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
      if (ov > best || (ov == best && oi < bi)) {
        best = ov;
        bi = oi;
      }
    }
    if (lane == 0) {
      wv[warp] = best;
      wi[warp] = bi;
    }
    __syncthreads();
    best = wv[0];
    bi = wi[0];
    const int nw = min(PANEL_THREADS / 32, (cnt + 31) / 32);  // warps that hold rows
    for (int w = 1; w < nw; ++w)
      if (wv[w] > best || (wv[w] == best && wi[w] < bi)) {
        best = wv[w];
        bi = wi[w];
      }
    if (tid < kb) {
      if (bi < n) {
        const double v = M[(bi - lo) * PANEL_PITCH + tid];
        for (int q = 0; q < csize; ++q) cl.map_shared_rank(&st, q)->from[rank].cand[tid] = v;
      }
    } else if (tid >= 64 && tid < 64 + kb) {
      if (r >= lo && r < lo + cnt) {
        const double v = M[(r - lo) * PANEL_PITCH + tid - 64];
        for (int q = 0; q < csize; ++q) cl.map_shared_rank(&st, q)->rrow[tid - 64] = v;
      }
    } else if (tid >= 128 && tid < 128 + csize) {
      PanelPub* o = &cl.map_shared_rank(&st, tid - 128)->from[rank];
      o->val = best;
      o->idx = bi;
    }
    cl.sync();
    int win = 0, p = n;
    long long pval = -2;
    for (int q = 0; q < csize; ++q) {
      const long long v = st.from[q].val;
      const int oi = st.from[q].idx;
      if (v > pval || (v == pval && oi < p)) {
        pval = v;
        p = oi;
        win = q;
      }
    }
    if (pval <= 0 || pval >= 0x7FF0000000000000ll) {  // zero or non-finite pivot (the same in every CTA)
      if (rank == 0) {
        if (tid == 0) atomicExch(status, int(LEM_ENUMERIC));
        for (int q = c + tid; q < kb; q += PANEL_THREADS) piv[b * GJ_KB + q] = k0 + q;  // no more swaps
      }
      break;
    }
    if (tid < kb) {
      const double inv = 1.0 / st.from[win].cand[c];
      prow[tid] = tid == c ? inv : st.from[win].cand[tid] * inv;
    } else if (tid >= 64 && tid < 64 + kb && p != r && p >= lo && p < lo + cnt) {
      const int q = tid - 64;
      const double old = st.rrow[q];
      M[(p - lo) * PANEL_PITCH + q] = old;
      if (q == c) {
        fcol[p - lo] = old;
        fzero[p - lo] = (__double_as_longlong(old) & 0x7FFFFFFFFFFFFFFFll) == 0;
      }
    }
    if (rank == 0 && tid == 128) piv[b * GJ_KB + c] = p;
    __syncthreads();
    if (j < kb) {
      const double pj = prow[j];
      constexpr int U = 4, ST = PANEL_THREADS / GJ_KB;  // rows in flight, row step
      auto upd = [&](double f, int zero, double m, int i) {
        const double v = fma(-f, pj, j == c ? 0.0 : m);
        return lo + i == r ? pj : zero ? m : v;
      };
      int i = grp;
      for (; i + (U - 1) * ST < cnt; i += U * ST) {
        double f[U], m[U];
        int z[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          f[u] = fcol[i + u * ST];
          z[u] = fzero[i + u * ST];
          m[u] = M[(i + u * ST) * PANEL_PITCH + j];
        }
#pragma unroll
        for (int u = 0; u < U; ++u) m[u] = upd(f[u], z[u], m[u], i + u * ST);
#pragma unroll
        for (int u = 0; u < U; ++u) M[(i + u * ST) * PANEL_PITCH + j] = m[u];
      }
#pragma unroll 1
      for (; i < cnt; i += ST) M[i * PANEL_PITCH + j] = upd(fcol[i], fzero[i], M[i * PANEL_PITCH + j], i);
    }
    __syncthreads();
  }
  cl.sync();  // no CTA leaves while another may write into its memory
  double* Yb = Y + int64_t(b) * n * GJ_KB;
  for (int e = tid; e < cnt * GJ_KB; e += PANEL_THREADS) {
    const int i = e / GJ_KB, q = e % GJ_KB;
    if (q < kb) Yb[int64_t(lo + i) * GJ_KB + q] = M[i * PANEL_PITCH + q];
  }
}

static cudaError_t launch_panel(const double* src, int64_t lds, int64_t ss, int n, int k0, int kb, double* Y,
                                int* piv, int* status, int nb, cudaStream_t st) {
  // 8 rows a CTA at least: panels of 64 rows took 167, 134 and 122 us on 2, 4 and 8 CTAs
  const int csize = std::min(PANEL_MAX_CLUSTER, (n + 7) / 8);
  const int rows_per = (n + csize - 1) / csize;
  const size_t smem = 2 * sizeof(PanelStep) + sizeof(double) * (size_t(rows_per) * (PANEL_PITCH + 2) + GJ_KB);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(unsigned(nb) * csize);
  cfg.blockDim = dim3(PANEL_THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = unsigned(csize);
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, bgj_panel_kernel, src, lds, ss, n, k0, kb, csize, rows_per, Y, piv, status);
}

// Row swaps k0 + c <-> piv[c], c < kb, in order, on columns [0, cols) of a matrix.
// rows (not null): the pivot rows k0 .. k0 + kb - 1 then move there (kb x cols), leaving zeros.
__global__ void bgj_swap_kernel(double* M, int64_t ld, int64_t stride, int cols, int k0, int kb, const int* piv,
                                double* rows) {
  const int b = blockIdx.y;
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= cols) return;
  double* m = M + int64_t(b) * stride + j;
  for (int c = 0; c < kb; ++c) {
    const int p = piv[b * GJ_KB + c];
    if (p == k0 + c) continue;
    const double a = m[int64_t(k0 + c) * ld];
    m[int64_t(k0 + c) * ld] = m[int64_t(p) * ld];
    m[int64_t(p) * ld] = a;
  }
  if (!rows) return;
  double* r = rows + int64_t(b) * kb * cols + j;
  for (int c = 0; c < kb; c += 16) {  // sixteen loads in flight
    double v[16];
#pragma unroll
    for (int u = 0; u < 16; ++u) v[u] = c + u < kb ? m[int64_t(k0 + c + u) * ld] : 0.0;
#pragma unroll
    for (int u = 0; u < 16; ++u)
      if (c + u < kb) {
        r[int64_t(c + u) * cols] = v[u];
        m[int64_t(k0 + c + u) * ld] = 0.0;
      }
  }
}

// rows of the owner tile D inside the window, from the squared result (n x n): R, or R1 for the
// matrices that `odd` marks (they stopped squaring an odd number of steps early)
__global__ void extract_rows_kernel(double* P, int64_t n_int, int64_t n_loc, const double* R0, const double* R1,
                                    const int* odd, int n, const BatchClass* bc) {
  const int b = blockIdx.y;
  const int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (e >= n_int * n_loc) return;
  const int i = int(e / n_loc), k = int(e % n_loc);
  const BatchClass c = bc[b];
  const int ie = c.rep.iext[0] * c.rep.iext[1];
  const int wl = c.rep.wext[0] * c.rep.wext[1];
  double v = 0.0;
  if (i < ie && k < wl && k < n) {
    const int row = (c.rep.iofs[0] + i / c.rep.iext[1]) * c.rep.wext[1] + c.rep.iofs[1] + i % c.rep.iext[1];
    v = (odd && odd[b] ? R1 : R0)[int64_t(b) * n * n + int64_t(row) * n + k];
  }
  P[int64_t(b) * n_int * n_loc + e] = v;
}

// Complex problems: owner rows of the embedded result R (n x n, n = 2 x window nodes) into P
// (n_int x n_loc, both embedded sizes): rows [0, n_int/2) the real parts, [n_int/2, n_int) the
// imaginary parts of the owner nodes; columns as in R (real parts, then imaginary parts).
__global__ void extract_rows_complex_kernel(double* P, int64_t n_int, int64_t n_loc, const double* R0,
                                            const double* R1, const int* odd, int n, const BatchClass* bc) {
  const int b = blockIdx.y;
  const int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (e >= n_int * n_loc) return;
  const int i = int(e / n_loc), k = int(e % n_loc);
  const int hi = int(n_int / 2), hn = n / 2;
  const int comp = i / hi, io = i % hi;
  const BatchClass c = bc[b];
  const int ie = c.rep.iext[0] * c.rep.iext[1];
  double v = 0.0;
  if (io < ie && k < n) {
    const int row = (c.rep.iofs[0] + io / c.rep.iext[1]) * c.rep.wext[1] + c.rep.iofs[1] + io % c.rep.iext[1];
    v = (odd && odd[b] ? R1 : R0)[int64_t(b) * n * n + int64_t(comp * hn + row) * n + k];
  }
  P[int64_t(b) * n_int * n_loc + e] = v;
}

__global__ void copy_cols_kernel(double* dst, int64_t ldd, int dcol0, const double* src, int64_t lds,
                                 int scol0, int n, int ncols) {
  const int b = blockIdx.y;
  const int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (e >= int64_t(n) * ncols) return;
  const int i = int(e / ncols), j = int(e % ncols);
  dst[int64_t(b) * n * ldd + int64_t(i) * ldd + dcol0 + j] = src[int64_t(b) * n * lds + int64_t(i) * lds + scol0 + j];
}

// Device scratch of one build batch, released when the batch is done. A context that rebuilds
// (refresh > 0) keeps one block of the size its builds took, up to kKeepBytes and kKeepAll over all
// contexts, and later batches are laid out in it: taking and returning gigabytes at the stream-ordered
// pool cost 5 ms of a 27 ms build, since the pool gives them back to the driver at every synchronisation.
// It is given back with the context, or when another allocation of the context finds no room. Otherwise
// each piece comes from cudaMallocAsync and is freed in the order of the build's stream: a build that
// fails half way leaves kernels in flight that still use it.
constexpr int64_t kKeepBytes = int64_t(4) << 30, kKeepAll = int64_t(16) << 30;
std::atomic<int64_t> g_kept{0};
struct Scratch {
  lem_ctx* ctx;
  size_t used = 0;
  std::vector<void*> own;
  explicit Scratch(lem_ctx* c) : ctx(c) {}
  Scratch(const Scratch&) = delete;
  Scratch& operator=(const Scratch&) = delete;
  lem_status get(void** p, size_t bytes) {
    const size_t b = (bytes + 255) / 256 * 256, o = used;
    used += b;
    if (used <= ctx->ws_bytes) {
      *p = static_cast<char*>(ctx->d_ws) + o;
      return LEM_OK;
    }
    if (fault_alloc(bytes)) return fail(LEM_ENOMEM, "build scratch refused (LEM_FAULT=alloc)");
    LEM_CUDA_TRY(cudaMallocAsync(p, b, ctx->stream));
    own.push_back(*p);
    return LEM_OK;
  }
  template <class T>
  lem_status get(T** p, size_t count) { return get(reinterpret_cast<void**>(p), sizeof(T) * count); }
  ~Scratch() {
    for (void* p : own) cudaFreeAsync(p, ctx->stream);
  }
  // after a build that went well
  void keep() {
    if (own.empty() || ctx->desc.refresh <= 0 || !ctx->desc.reaction || int64_t(used) > kKeepBytes) return;
    for (void* p : own) cudaFreeAsync(p, ctx->stream);
    own.clear();
    builder_release(ctx);
    if (g_kept.fetch_add(int64_t(used)) + int64_t(used) > kKeepAll || dev_alloc(ctx, &ctx->d_ws, used) != LEM_OK)
      g_kept -= int64_t(used);
    else
      ctx->ws_bytes = used;
  }
};

inline dim3 grid1(int64_t total, int by) { return dim3(unsigned((total + 255) / 256), by); }

}  // namespace

void builder_release(lem_ctx* ctx) {
  if (!ctx->d_ws) return;
  cudaFreeAsync(ctx->d_ws, ctx->stream);
  ctx->d_ws = nullptr;
  ctx->device_bytes -= int64_t(ctx->ws_bytes);
  g_kept -= int64_t(ctx->ws_bytes);
  ctx->ws_bytes = 0;
}

bool builder_uses_tc(int prec) {
  if (prec == LEM_PREC_FP64) return false;
  const char* e = std::getenv("LEM_BUILD_PRODUCTS");  // "fp64": FP64 products in every tier
  return !(e && std::string(e) == "fp64");
}

namespace {
struct TcGuard {
  TcGemm* g = nullptr;
  ~TcGuard() { tc_gemm_destroy(g); }
};
}  // namespace

// One A against a list of right factors, on the tensor cores (tcg not null) or in FP64.
static lem_status mul_list(lem_ctx* ctx, TcGemm* tcg, int nbatch, const int* map, int M, int K, const double* A,
                           int64_t lda, int64_t sA, const TcProduct* list, int np, int zr0, int zr1) {
  if (tcg) return tc_gemm(tcg, nbatch, map, M, K, A, lda, sA, list, np, zr0, zr1, ctx->stream);
  DgemmList g{};
  g.M = M; g.K = K; g.np = np; g.A = A; g.lda = lda; g.sA = sA; g.map = map;
  for (int t = 0; t < np; ++t) {
    const TcProduct& p = list[t];
    g.N[t] = p.N;
    g.B[t] = p.B; g.ldb[t] = p.ldb; g.sB[t] = p.sB;
    g.D[t] = p.D; g.ldd[t] = p.ldd; g.sD[t] = p.sD;
    g.C[t] = p.C; g.ldc[t] = p.ldc; g.sC[t] = p.sC;
    g.diag[t] = p.diag;
  }
  int nsm = 0;
  if (cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, ctx->device) != cudaSuccess || nsm < 1) nsm = 152;
  LEM_CUDA_TRY(dgemm_list(g, nbatch, nsm, ctx->stream));
  return LEM_OK;
}

// Gauss-Jordan elimination of G = [Q | RHS] (nb matrices of n x gjcols): on exit the RHS
// columns hold Q^{-1} RHS. Panels in FP64, the other columns by products (tcg: on tcgen05).
static lem_status solve_gj(lem_ctx* ctx, TcGemm* tcg, double* G, int n, int gjcols, int nb, Scratch& ws) {
  cudaStream_t st = ctx->stream;
  double *Y = nullptr, *rows = nullptr;
  int* piv = nullptr;
  LEM_TRY(ws.get(&Y, size_t(nb) * n * GJ_KB));
  LEM_TRY(ws.get(&piv, size_t(nb) * GJ_KB));
  // FP64 products write over their right factor: the pivot rows move out first
  if (!tcg) LEM_TRY(ws.get(&rows, size_t(nb) * GJ_KB * gjcols));
  LEM_CUDA_TRY(allow_smem(reinterpret_cast<const void*>(bgj_panel_kernel), ctx->device, 0, 1024));
  const int64_t sG = int64_t(n) * gjcols, sY = int64_t(n) * GJ_KB;
  for (int k0 = 0; k0 < n; k0 += GJ_KB) {  // a panel of columns
    const int kb = std::min(GJ_KB, n - k0);
    if (n <= PANEL_MAX_N) {
      LEM_CUDA_TRY(launch_panel(G + k0, gjcols, sG, n, k0, kb, Y, piv, ctx->d_status, nb, st));
    } else {
      copy_cols_kernel<<<grid1(int64_t(n) * kb, nb), 256, 0, st>>>(Y, GJ_KB, 0, G, gjcols, k0, n, kb);
      for (int c = 0; c < kb; ++c) {
        bgj_pivot_kernel<<<nb, 256, 0, st>>>(Y, n, k0, c, kb, piv, ctx->d_status);
        bgj_elim_kernel<<<dim3((n + 3) / 4, nb), 256, 0, st>>>(Y, n, k0, c, kb);
      }
    }
    // the columns behind the panel: C = Y B + D with B the pivot rows, D without them
    const int m_r = gjcols - (k0 + kb);
    double* T = G + (k0 + kb);
    bgj_swap_kernel<<<dim3((m_r + 255) / 256, nb), 256, 0, st>>>(T, gjcols, sG, m_r, k0, kb, piv, rows);
    LEM_CUDA_TRY(cudaGetLastError());
    const double* B = tcg ? T + int64_t(k0) * gjcols : rows;
    const TcProduct pr{m_r, B, tcg ? gjcols : m_r, tcg ? sG : int64_t(kb) * m_r, T, gjcols, sG, T, gjcols, sG, nullptr};
    LEM_TRY(mul_list(ctx, tcg, nb, nullptr, n, kb, Y, GJ_KB, sY, &pr, 1, k0, k0 + kb));
  }
  LEM_CUDA_TRY(cudaGetLastError());
  return LEM_OK;
}

// Build the propagators of classes [c0, c0 + nb) into P (nb x n_int x n_loc).
static lem_status build_batch(lem_ctx* ctx, int c0, int nb, const double* d_state) {
  cudaStream_t st = ctx->stream;
  const int n = int(ctx->n_loc);
  const bool phi = ctx->desc.mode == LEM_MODE_PHI;
  const int64_t nn = int64_t(n) * n;
  std::vector<BatchClass> hbc(nb);
  for (int b = 0; b < nb; ++b) {
    const ClassDesc& c = ctx->classes[c0 + b];
    hbc[b].rep = ctx->tiles[c.rep_tile];
    hbc[b].whole[0] = c.whole[0];
    hbc[b].whole[1] = c.whole[1];
  }
  // device scratch for this batch (freed at return)
  const int nmat = phi ? 15 : 9;
  const int gjcols = phi ? 3 * n : 2 * n;
  Scratch ws(ctx);
  double *S = nullptr, *d_norm = nullptr, *d_c = nullptr;
  BatchClass* d_bc = nullptr;
  int* d_map = nullptr;
  LEM_TRY(ws.get(&S, (size_t(nmat) * nn + size_t(n) * gjcols) * nb));
  LEM_TRY(ws.get(&d_bc, size_t(nb)));
  LEM_TRY(ws.get(&d_norm, size_t(nb)));
  LEM_TRY(ws.get(&d_c, size_t(2) * nb));
  LEM_TRY(ws.get(&d_map, size_t(2) * nb));
  LEM_CUDA_TRY(cudaMemcpyAsync(d_bc, hbc.data(), sizeof(BatchClass) * nb, cudaMemcpyHostToDevice, st));
  auto M = [&](int i) { return S + size_t(i) * nn * nb; };
  double *Xs = M(0), *T2 = M(1), *T4 = M(2), *T6 = M(3), *TW = M(4), *TV = M(5), *T3 = M(6), *VT = M(7), *UT = M(8);
  double *B2 = nullptr, *B4 = nullptr, *B6 = nullptr, *BW = nullptr, *B3 = nullptr, *UB = nullptr;
  if (phi) { B2 = M(9); B4 = M(10); B6 = M(11); BW = M(12); B3 = M(13); UB = M(14); }
  double* G = S + size_t(nmat) * nn * nb;  // n x gjcols per batch entry

  // X = dt A_M (+ reaction Jacobian)
  const double* u = ctx->desc.reaction ? d_state : nullptr;
  LEM_CUDA_TRY(cudaMemsetAsync(Xs, 0, sizeof(double) * nn * nb, st));
  if (ctx->cplx)  // the real embedding of the complex window matrix
    assemble_local_complex_kernel<<<dim3((n / 2 + 127) / 128, nb), 128, 0, st>>>(
        Xs, n, d_bc, nb, ctx->d_coef, ctx->desc.coef_stride, ctx->ny, ctx->nx, ctx->desc.ndim);
  else
    assemble_local_kernel<<<dim3((n + 127) / 128, nb), 128, 0, st>>>(
        Xs, n, d_bc, nb, ctx->d_coef, ctx->desc.coef_stride, ctx->ny, ctx->nx, ctx->desc.ndim, u,
        ctx->desc.dt, ctx->desc.reaction, ctx->desc.porous_m);
  LEM_CUDA_TRY(cudaGetLastError());
  // exact 1-norms -> s per class (host decides, same rule as theta_13 scaling)
  LEM_CUDA_TRY(cudaMemsetAsync(d_norm, 0, sizeof(double) * nb, st));
  norm1_kernel<<<dim3((n + 31) / 32, nb), 256, 0, st>>>(
      Xs, n, reinterpret_cast<unsigned long long*>(d_norm));
  LEM_CUDA_TRY(cudaGetLastError());
  std::vector<double> norms(nb), scales(2 * nb);
  LEM_CUDA_TRY(cudaMemcpyAsync(norms.data(), d_norm, sizeof(double) * nb, cudaMemcpyDeviceToHost, st));
  LEM_CUDA_TRY(cudaStreamSynchronize(st));
  std::vector<int> s(nb);
  int smax = 0;
  for (int b = 0; b < nb; ++b) {
    double nz = phi ? std::max(norms[b], 1.0) : norms[b];  // ||[[X, I], [0, 0]]||_1
    int sb = 0;
    while (nz > kTheta13 * std::ldexp(1.0, sb)) ++sb;
    s[b] = sb;
    smax = std::max(smax, sb);
    ctx->squarings[c0 + b] = sb;
    scales[b] = std::ldexp(1.0, -sb);                       // c = 2^-s
    scales[nb + b] = std::ldexp(1.0, -sb) * (kPadeInt[1] / kPadeInt[0]);  // c * b1
  }
  double* d_cb1 = d_c + nb;
  LEM_CUDA_TRY(cudaMemcpyAsync(d_c, scales.data(), sizeof(double) * 2 * nb, cudaMemcpyHostToDevice, st));
  // Classes sorted by s, descending: at squaring q the classes still squaring (s > q) are a
  // prefix of the order, so one index map serves every squaring. A class that stops an odd
  // number of squarings early has its result in the other buffer of the pair.
  std::vector<int> order(2 * nb);
  std::iota(order.begin(), order.begin() + nb, 0);
  std::stable_sort(order.begin(), order.begin() + nb, [&](int a, int b) { return s[a] > s[b]; });
  for (int b = 0; b < nb; ++b) order[nb + b] = (smax - s[b]) & 1;
  const int* d_odd = d_map + nb;
  LEM_CUDA_TRY(cudaMemcpyAsync(d_map, order.data(), sizeof(int) * 2 * nb, cudaMemcpyHostToDevice, st));

  PadeTerms pt{};
  for (int j = 0; j < 14; ++j) pt.b[j] = kPadeInt[j] / kPadeInt[0];
  const dim3 gsq = grid1(nn, nb);
  TcGuard tc;
  if (ctx->build_tc) {
    char* mem = nullptr;
    LEM_TRY(ws.get(&mem, tc_gemm_bytes(n, nb, gjcols, phi ? 4 : 2)));
    LEM_TRY(tc_gemm_create(n, nb, gjcols, phi ? 4 : 2, mem, st, &tc.g));
  }
  // C = A B (+ D, which may be C) (+ diag I) for every product of the list, on the first nact
  // classes of the order (nact == nb: all)
  struct Term { const double* B; const double* D; double* C; const double* diag; };
  auto mul = [&](int nact, const double* A, std::initializer_list<Term> list) -> lem_status {
    TcProduct pr[4];
    int np = 0;
    for (const Term& t : list) pr[np++] = TcProduct{n, t.B, n, nn, t.D, n, nn, t.C, n, nn, t.diag};
    return mul_list(ctx, tc.g, nact, nact == nb ? nullptr : d_map, n, n, A, n, nn, pr, np, 0, 0);
  };
  // Xs = X / 2^s (per class), Z^2's top-right c Xs; then the powers
  scale_kernel<<<gsq, 256, 0, st>>>(Xs, B2, nn, d_c);
  LEM_CUDA_TRY(cudaGetLastError());
  LEM_TRY(mul(nb, Xs, {{Xs, nullptr, T2, nullptr}}));
  if (phi) {
    LEM_TRY(mul(nb, T2, {{T2, nullptr, T4, nullptr}, {B2, nullptr, B4, nullptr}}));
    LEM_TRY(mul(nb, T4, {{T2, nullptr, T6, nullptr}, {B2, nullptr, B6, nullptr}}));
  } else {
    LEM_TRY(mul(nb, T2, {{T2, nullptr, T4, nullptr}}));
    LEM_TRY(mul(nb, T4, {{T2, nullptr, T6, nullptr}}));
  }
  // W1 = b13 Z6 + b11 Z4 + b9 Z2 ;  W3 = Z6 W1 + b7 Z6 + b5 Z4 + b3 Z2 + b1 I ; U = Z W3
  // V = Z6 (b12 Z6 + b10 Z4 + b8 Z2) + b6 Z6 + b4 Z4 + b2 Z2 + b0 I
  pt.z2[0] = T2; pt.z4[0] = T4; pt.z6[0] = T6; pt.w[0] = TW; pt.v[0] = TV; pt.a3[0] = T3; pt.vt[0] = VT;
  pt.z2[1] = B2; pt.z4[1] = B4; pt.z6[1] = B6; pt.w[1] = BW; pt.a3[1] = B3;
  pade_terms_kernel<<<dim3(unsigned((nn * nb + 255) / 256), 1, phi ? 2 : 1), 256, 0, st>>>(pt, n, nn * nb);
  LEM_CUDA_TRY(cudaGetLastError());
  if (phi) {
    LEM_TRY(mul(nb, T6, {{TW, T3, T3, nullptr}, {BW, B3, B3, nullptr}, {TV, VT, VT, nullptr}}));
    // UB = X B3 + c b1 I (Z's top-right c I times b1); V_B + U_B - (V_B - U_B) = 2 U_B: V_B drops out
    LEM_TRY(mul(nb, Xs, {{T3, nullptr, UT, nullptr}, {B3, nullptr, UB, d_cb1}}));
  } else {
    LEM_TRY(mul(nb, T6, {{TW, T3, T3, nullptr}, {TV, VT, VT, nullptr}}));
    LEM_TRY(mul(nb, Xs, {{T3, nullptr, UT, nullptr}}));
  }
  // G = [V_T - U_T | V_T + U_T | (V_B + U_B) - (V_B - U_B) = 2 U_B]
  solve_system_kernel<<<gsq, 256, 0, st>>>(G, n, gjcols, VT, UT, UB);
  LEM_CUDA_TRY(cudaGetLastError());
  LEM_CUDA_TRY(cudaMemsetAsync(ctx->d_status, 0, sizeof(int), st));
  LEM_TRY(solve_gj(ctx, tc.g, G, n, gjcols, nb, ws));
  LEM_CUDA_TRY(cudaGetLastError());
  // R_T and R_B, then the squarings (R_T, R_B)^2 = (R_T^2, R_T R_B + R_B)
  double *RT = T2, *RTn = T4, *RB = B2, *RBn = B4;
  copy_cols_kernel<<<gsq, 256, 0, st>>>(RT, n, 0, G, gjcols, n, n, n);
  if (phi) copy_cols_kernel<<<gsq, 256, 0, st>>>(RB, n, 0, G, gjcols, 2 * n, n, n);
  LEM_CUDA_TRY(cudaGetLastError());
  for (int q = 0; q < smax; ++q) {
    int nact = 0;
    while (nact < nb && s[order[nact]] > q) ++nact;
    if (!phi)
      LEM_TRY(mul(nact, RT, {{RT, nullptr, RTn, nullptr}}));
    else if (q == smax - 1)  // phi_1 is R_B: the last R_T^2 is not needed
      LEM_TRY(mul(nact, RT, {{RB, RB, RBn, nullptr}}));
    else
      LEM_TRY(mul(nact, RT, {{RB, RB, RBn, nullptr}, {RT, nullptr, RTn, nullptr}}));
    std::swap(RT, RTn);
    if (phi) std::swap(RB, RBn);
  }
  const double* R = phi ? RB : RT;
  const double* R1 = phi ? RBn : RTn;
  double* Pout = ctx->d_P + size_t(c0) * ctx->n_int * ctx->n_loc;
  if (ctx->cplx)
    extract_rows_complex_kernel<<<grid1(ctx->n_int * ctx->n_loc, nb), 256, 0, st>>>(Pout, ctx->n_int, ctx->n_loc, R,
                                                                                    R1, d_odd, n, d_bc);
  else
    extract_rows_kernel<<<grid1(ctx->n_int * ctx->n_loc, nb), 256, 0, st>>>(Pout, ctx->n_int, ctx->n_loc, R, R1, d_odd,
                                                                            n, d_bc);
  LEM_CUDA_TRY(cudaGetLastError());
  int status = 0;
  LEM_CUDA_TRY(cudaMemcpyAsync(&status, ctx->d_status, sizeof(int), cudaMemcpyDeviceToHost, st));
  LEM_CUDA_TRY(cudaStreamSynchronize(st));
  if (status != 0) return fail(LEM_ENUMERIC, "singular Pade denominator (V - U) in the propagator build");
  if (tc.g) LEM_TRY(tc_gemm_check(tc.g, st));
  ws.keep();
  return LEM_OK;
}

// ---------------------------------------------------------------- phi_1 and phi_3 together
// For the third-order Rosenbrock step each class needs phi_1(X) and phi_3(X). Both are blocks
// of exp(Z), Z = [[X, I, 0, 0], [0, 0, I, 0], [0, 0, 0, I], [0, 0, 0, 0]] (top block row:
// e^X, phi_1, phi_2, phi_3). Every polynomial in Z, and its inverse, has the form
//   [[T, B0, B1, B2], [0, b0 I, b1 I, b2 I], [0, 0, b0 I, b1 I], [0, 0, 0, b0 I]]
// (an "augmented" element: T and B_j n x n, b a scalar upper-triangular Toeplitz part), with
//   (A C).T = A.T C.T,  (A C).B_j = A.T C.B_j + sum_{a <= j} c.b_{j-a} A.B_a,  b = a.b * c.b.
// The scaling is moved onto the functions: with Xs = X / 2^s, the Pade-13 approximant runs on
// Z(Xs) (unit identity blocks, so every weight and the Toeplitz parts are the same for every
// class), and s doublings 2^k phi_k(2Y) = e^Y phi_k(Y) + sum_{j=1..k} phi_j(Y) / (k - j)!
// bring phi_k(Xs) back to phi_k(X). s follows the same rule as the phi_1 build (the 1-norm of
// the augmented matrix is max(|X|_1, 1)).
struct Aug {
  double* m[4];  // T, B0, B1, B2
  double b[3];   // Toeplitz part (class independent)
};

static lem_status build_batch_phi3(lem_ctx* ctx, int c0, int nb, const double* d_state) {
  cudaStream_t st = ctx->stream;
  const int n = int(ctx->n_loc);
  const int64_t nn = int64_t(n) * n;
  std::vector<BatchClass> hbc(nb);
  for (int b = 0; b < nb; ++b) {
    const ClassDesc& c = ctx->classes[c0 + b];
    hbc[b].rep = ctx->tiles[c.rep_tile];
    hbc[b].whole[0] = c.whole[0];
    hbc[b].whole[1] = c.whole[1];
  }
  constexpr int NAUG = 10;  // Z, Z2, Z4, Z6, W, W3, U, V, R, Rn
  const int gjcols = 5 * n;
  Scratch ws(ctx);
  double *S = nullptr, *d_norm = nullptr, *d_scale = nullptr;
  BatchClass* d_bc = nullptr;
  int* d_map = nullptr;
  LEM_TRY(ws.get(&S, (size_t(NAUG) * 4 * nn + size_t(n) * gjcols) * nb));
  LEM_TRY(ws.get(&d_bc, size_t(nb)));
  LEM_TRY(ws.get(&d_norm, size_t(nb)));
  LEM_TRY(ws.get(&d_scale, size_t(nb)));
  LEM_TRY(ws.get(&d_map, size_t(2) * nb));
  LEM_CUDA_TRY(cudaMemcpyAsync(d_bc, hbc.data(), sizeof(BatchClass) * nb, cudaMemcpyHostToDevice, st));
  auto aug = [&](int i) {
    Aug a;
    for (int q = 0; q < 4; ++q) a.m[q] = S + (size_t(i) * 4 + q) * nn * nb;
    a.b[0] = a.b[1] = a.b[2] = 0.0;
    return a;
  };
  Aug Z = aug(0), Z2 = aug(1), Z4 = aug(2), Z6 = aug(3), W = aug(4), W3 = aug(5), U = aug(6), V = aug(7),
      R = aug(8), Rn = aug(9);
  double* G = S + size_t(NAUG) * 4 * nn * nb;

  // X = dt J_M, the 1-norms, s per class
  const double* u = ctx->desc.reaction ? d_state : nullptr;
  LEM_CUDA_TRY(cudaMemsetAsync(Z.m[0], 0, sizeof(double) * nn * nb, st));
  assemble_local_kernel<<<dim3((n + 127) / 128, nb), 128, 0, st>>>(
      Z.m[0], n, d_bc, nb, ctx->d_coef, ctx->desc.coef_stride, ctx->ny, ctx->nx, ctx->desc.ndim, u, ctx->desc.dt,
      ctx->desc.reaction, ctx->desc.porous_m);
  LEM_CUDA_TRY(cudaMemsetAsync(d_norm, 0, sizeof(double) * nb, st));
  norm1_kernel<<<dim3((n + 31) / 32, nb), 256, 0, st>>>(Z.m[0], n,
                                                           reinterpret_cast<unsigned long long*>(d_norm));
  LEM_CUDA_TRY(cudaGetLastError());
  std::vector<double> norms(nb), scales(nb);
  LEM_CUDA_TRY(cudaMemcpyAsync(norms.data(), d_norm, sizeof(double) * nb, cudaMemcpyDeviceToHost, st));
  LEM_CUDA_TRY(cudaStreamSynchronize(st));
  std::vector<int> s(nb);
  int smax = 0;
  for (int b = 0; b < nb; ++b) {
    const double nz = std::max(norms[b], 1.0);
    int sb = 0;
    while (nz > kTheta13 * std::ldexp(1.0, sb)) ++sb;
    s[b] = sb;
    smax = std::max(smax, sb);
    ctx->squarings[c0 + b] = sb;
    scales[b] = std::ldexp(1.0, -sb);
  }
  LEM_CUDA_TRY(cudaMemcpyAsync(d_scale, scales.data(), sizeof(double) * nb, cudaMemcpyHostToDevice, st));

  const dim3 gsq = grid1(nn, nb);
  auto lin = [&](double* out, std::initializer_list<std::pair<const double*, double>> terms, double diag,
                 const double* wscale0) -> lem_status {
    Lin L{};
    L.nin = 0;
    for (auto& t : terms) {
      if (t.second == 0.0) continue;  // never read a buffer that is not needed (it may be unset)
      L.in[L.nin] = t.first;
      L.w[L.nin] = t.second;
      ++L.nin;
    }
    L.diag = diag;
    L.dscale = nullptr;
    L.wscale0 = wscale0;
    lincomb_kernel<<<gsq, 256, 0, st>>>(out, n, n, n, L);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? LEM_OK : cuda_fail(e, "lincomb_kernel");
  };
  TcGuard tc;
  if (ctx->build_tc) {
    char* mem = nullptr;
    LEM_TRY(ws.get(&mem, tc_gemm_bytes(n, nb, gjcols, 4)));
    LEM_TRY(tc_gemm_create(n, nb, gjcols, 4, mem, st, &tc.g));
  }
  // one A against four B
  auto mul4 = [&](int nact, const int* map, const double* A, const double* const (&B)[4], const double* const (&D)[4],
                  double* const (&C)[4]) -> lem_status {
    TcProduct pr[4];
    for (int t = 0; t < 4; ++t) pr[t] = TcProduct{n, B[t], n, nn, D[t], n, nn, C[t], n, nn, nullptr};
    return mul_list(ctx, tc.g, nact, map, n, n, A, n, nn, pr, 4, 0, 0);
  };
  // C = A * B (C distinct from A and B)
  auto amul = [&](const Aug& A, const Aug& B, Aug& C) -> lem_status {
    LEM_TRY(mul4(nb, nullptr, A.m[0], {B.m[0], B.m[1], B.m[2], B.m[3]}, {}, C.m));
    for (int j = 0; j < 3; ++j) {
      const double w0 = B.b[j], w1 = j >= 1 ? B.b[j - 1] : 0.0, w2 = j >= 2 ? B.b[j - 2] : 0.0;
      if (w0 != 0.0 || w1 != 0.0 || w2 != 0.0)  // + sum_{a <= j} B.b[j - a] A.B_a
        LEM_TRY(lin(C.m[1 + j], {{C.m[1 + j], 1.0}, {A.m[1], w0}, {A.m[2], w1}, {A.m[3], w2}}, 0.0, nullptr));
    }
    for (int j = 0; j < 3; ++j) {
      double v = 0.0;
      for (int a = 0; a <= j; ++a) v += A.b[a] * B.b[j - a];
      C.b[j] = v;
    }
    return LEM_OK;
  };
  // C = sum w_i A_i + d I (C may be one of the A_i)
  auto alin = [&](Aug& C, std::initializer_list<std::pair<const Aug*, double>> terms, double d) -> lem_status {
    double nb3[3] = {d, 0.0, 0.0};
    for (int q = 0; q < 4; ++q) {
      Lin L{};
      L.nin = 0;
      for (auto& t : terms) {
        L.in[L.nin] = t.first->m[q];
        L.w[L.nin] = t.second;
        ++L.nin;
      }
      L.diag = q == 0 ? d : 0.0;
      lincomb_kernel<<<gsq, 256, 0, st>>>(C.m[q], n, n, n, L);
    }
    LEM_CUDA_TRY(cudaGetLastError());
    for (auto& t : terms)
      for (int j = 0; j < 3; ++j) nb3[j] += t.second * t.first->b[j];
    for (int j = 0; j < 3; ++j) C.b[j] = nb3[j];
    return LEM_OK;
  };

  // Z(Xs): T = X / 2^s, B = (I, 0, 0), Toeplitz part N (b = (0, 1, 0))
  LEM_TRY(lin(Z.m[0], {{Z.m[0], 1.0}}, 0.0, d_scale));
  LEM_TRY(lin(Z.m[1], {}, 1.0, nullptr));
  LEM_CUDA_TRY(cudaMemsetAsync(Z.m[2], 0, sizeof(double) * nn * nb, st));
  LEM_CUDA_TRY(cudaMemsetAsync(Z.m[3], 0, sizeof(double) * nn * nb, st));
  Z.b[0] = 0.0; Z.b[1] = 1.0; Z.b[2] = 0.0;
  double bj[14];
  for (int j = 0; j < 14; ++j) bj[j] = kPadeInt[j] / kPadeInt[0];
  LEM_TRY(amul(Z, Z, Z2));
  LEM_TRY(amul(Z2, Z2, Z4));
  LEM_TRY(amul(Z4, Z2, Z6));
  // U = Z (Z6 (b13 Z6 + b11 Z4 + b9 Z2) + b7 Z6 + b5 Z4 + b3 Z2 + b1 I)
  LEM_TRY(alin(W, {{&Z6, bj[13]}, {&Z4, bj[11]}, {&Z2, bj[9]}}, 0.0));
  LEM_TRY(amul(Z6, W, W3));
  LEM_TRY(alin(W3, {{&W3, 1.0}, {&Z6, bj[7]}, {&Z4, bj[5]}, {&Z2, bj[3]}}, bj[1]));
  LEM_TRY(amul(Z, W3, U));
  // V = Z6 (b12 Z6 + b10 Z4 + b8 Z2) + b6 Z6 + b4 Z4 + b2 Z2 + b0 I
  LEM_TRY(alin(W, {{&Z6, bj[12]}, {&Z4, bj[10]}, {&Z2, bj[8]}}, 0.0));
  LEM_TRY(amul(Z6, W, V));
  LEM_TRY(alin(V, {{&V, 1.0}, {&Z6, bj[6]}, {&Z4, bj[4]}, {&Z2, bj[2]}}, bj[0]));
  // R = (V - U)^{-1} (V + U). With M = V - U = [[Ma, Mc], [0, Md]] and P = V + U likewise:
  // R.T = Ma^{-1} Pa, R.B = Ma^{-1} (Pc - Mc g), g = Md^{-1} Pd (a Toeplitz solve).
  LEM_TRY(alin(W, {{&V, 1.0}, {&U, -1.0}}, 0.0));   // M
  LEM_TRY(alin(W3, {{&V, 1.0}, {&U, 1.0}}, 0.0));   // P
  double g[3];
  g[0] = W3.b[0] / W.b[0];
  g[1] = (W3.b[1] - W.b[1] * g[0]) / W.b[0];
  g[2] = (W3.b[2] - W.b[1] * g[1] - W.b[2] * g[0]) / W.b[0];
  for (int j = 0; j < 3; ++j) {  // Pc_j - sum_{a <= j} Mc_a g_{j-a}
    const double w0 = g[j], w1 = j >= 1 ? g[j - 1] : 0.0, w2 = j >= 2 ? g[j - 2] : 0.0;
    LEM_TRY(lin(W3.m[1 + j], {{W3.m[1 + j], 1.0}, {W.m[1], -w0}, {W.m[2], -w1}, {W.m[3], -w2}}, 0.0, nullptr));
  }
  copy_cols_kernel<<<gsq, 256, 0, st>>>(G, gjcols, 0, W.m[0], n, 0, n, n);
  for (int q = 0; q < 4; ++q) copy_cols_kernel<<<gsq, 256, 0, st>>>(G, gjcols, (1 + q) * n, W3.m[q], n, 0, n, n);
  LEM_CUDA_TRY(cudaGetLastError());
  LEM_CUDA_TRY(cudaMemsetAsync(ctx->d_status, 0, sizeof(int), st));
  LEM_TRY(solve_gj(ctx, tc.g, G, n, gjcols, nb, ws));
  for (int q = 0; q < 4; ++q) copy_cols_kernel<<<gsq, 256, 0, st>>>(R.m[q], n, 0, G, gjcols, (1 + q) * n, n, n);
  LEM_CUDA_TRY(cudaGetLastError());

  // s doublings of (E, phi_1, phi_2, phi_3) per class. The scaled copies H_k = phi_k / 2^k and
  // the addends D_k go to free scratch first, then phi_k' = E H_k + D_k and E' = E E.
  double* H1 = Z2.m[0]; double* H2 = Z2.m[1]; double* H3 = Z2.m[2];
  double* D2 = Z4.m[0]; double* D3 = Z4.m[1];
  auto prep = [&](const Aug& X) -> lem_status {  // on every class (harmless for finished ones)
    LEM_TRY(lin(H1, {{X.m[1], 0.5}}, 0.0, nullptr));
    LEM_TRY(lin(H2, {{X.m[2], 0.25}}, 0.0, nullptr));
    LEM_TRY(lin(H3, {{X.m[3], 0.125}}, 0.0, nullptr));
    LEM_TRY(lin(D2, {{X.m[1], 0.25}, {X.m[2], 0.25}}, 0.0, nullptr));
    LEM_TRY(lin(D3, {{X.m[1], 0.0625}, {X.m[2], 0.125}, {X.m[3], 0.125}}, 0.0, nullptr));
    return LEM_OK;
  };
  std::vector<int> order(nb);
  std::iota(order.begin(), order.end(), 0);
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return s[a] > s[b]; });
  // classes that stop squaring an odd number of steps early have their result in the other buffer
  order.resize(2 * nb);
  for (int b = 0; b < nb; ++b) order[nb + b] = (smax - s[b]) & 1;
  LEM_CUDA_TRY(cudaMemcpyAsync(d_map, order.data(), sizeof(int) * 2 * nb, cudaMemcpyHostToDevice, st));
  const int* d_odd = d_map + nb;
  for (int q = 0; q < smax; ++q) {
    int nact = 0;
    while (nact < nb && s[order[nact]] > q) ++nact;
    LEM_TRY(prep(R));
    LEM_TRY(mul4(nact, nact == nb ? nullptr : d_map, R.m[0], {R.m[0], H1, H2, H3}, {nullptr, H1, D2, D3}, Rn.m));
    std::swap(R, Rn);
  }
  const size_t pc = size_t(ctx->n_int) * ctx->n_loc;
  extract_rows_kernel<<<grid1(ctx->n_int * ctx->n_loc, nb), 256, 0, st>>>(ctx->d_P + size_t(c0) * pc, ctx->n_int,
                                                                         ctx->n_loc, R.m[1], Rn.m[1], d_odd, n, d_bc);
  extract_rows_kernel<<<grid1(ctx->n_int * ctx->n_loc, nb), 256, 0, st>>>(ctx->d_P3 + size_t(c0) * pc, ctx->n_int,
                                                                         ctx->n_loc, R.m[3], Rn.m[3], d_odd, n, d_bc);
  LEM_CUDA_TRY(cudaGetLastError());
  int status = 0;
  LEM_CUDA_TRY(cudaMemcpyAsync(&status, ctx->d_status, sizeof(int), cudaMemcpyDeviceToHost, st));
  LEM_CUDA_TRY(cudaStreamSynchronize(st));
  if (status != 0) return fail(LEM_ENUMERIC, "singular Pade denominator (V - U) in the propagator build");
  if (tc.g) LEM_TRY(tc_gemm_check(tc.g, st));
  ws.keep();
  return LEM_OK;
}

lem_status build_propagators_impl(lem_ctx* ctx, const double* d_state);

lem_status build_propagators(lem_ctx* ctx, const double* d_state) {
  nvtxRangePushA("lem_build_propagators");
  const lem_status st = build_propagators_impl(ctx, d_state);
  nvtxRangePop();
  return st;
}

lem_status build_propagators_impl(lem_ctx* ctx, const double* d_state) {
  if (ctx->desc.reaction && !d_state) return fail(LEM_EINVAL, "the reaction Jacobian needs the state");
  const int64_t nc = int64_t(ctx->classes.size());
  const int64_t n = ctx->n_loc;
  const bool rb3 = ctx->desc.scheme == LEM_SCHEME_RB3;
  const int nmat = rb3 ? 45 : ctx->desc.mode == LEM_MODE_PHI ? 18 : 11;
  // batch size from a scratch budget of 8 GiB
  const int gjc = rb3 ? 5 * int(n) : ctx->desc.mode == LEM_MODE_PHI ? 3 * int(n) : 2 * int(n);
  const double per = double(nmat) * n * n * sizeof(double) +
                     (ctx->build_tc ? double(tc_gemm_bytes(int(n), 1, gjc, ctx->desc.mode == LEM_MODE_PHI ? 4 : 2)) + sizeof(double) * n * GJ_KB : sizeof(double) * (double(n) * GJ_KB + double(gjc) * GJ_KB));
  int64_t bmax = std::max<int64_t>(1, int64_t((8.0 * (1ull << 30)) / per));
  bmax = std::min<int64_t>(bmax, 65535);
  for (int64_t c0 = 0; c0 < nc; c0 += bmax) {
    int nb = int(std::min<int64_t>(bmax, nc - c0));
    LEM_TRY(rb3 ? build_batch_phi3(ctx, int(c0), nb, d_state) : build_batch(ctx, int(c0), nb, d_state));
  }
  // the third-order Rosenbrock step evaluates its defect with the Jacobian's state
  if (rb3 && ctx->desc.reaction)
    LEM_CUDA_TRY(cudaMemcpyAsync(ctx->d_um, d_state, sizeof(double) * ctx->npts, cudaMemcpyDeviceToDevice,
                                 ctx->stream));
  LEM_TRY(oz_pack(ctx));
  if (ctx->oz) LEM_CUDA_TRY(cudaStreamSynchronize(ctx->stream));
  ctx->built = true;
  ctx->build_gen++;
  ctx->steps_since_build = 0;
  return LEM_OK;
}

}  // namespace lem
