// Per-tile propagator application (Sec. 3 steps 1-3, Eq. lem) as one batched GEMV launch:
// one CTA per owner tile gathers the tile's window of the residual (or of the state in EXP
// mode) into shared memory, its warps stream the rows of the tile's propagator, and every
// row's result is written straight into its owner node (u_D += y, or u_D = y in EXP mode).
// The launch is bound by the propagator bytes in HBM (n_int x n_loc per tile), so the
// reduced-precision variant stores propagators in FP32 (half the bytes) and accumulates the
// products in float-float (complex rows: per-chunk FMA sums); the FP64 variant is the plain
// reference arithmetic.
//
// Jacobi update: all tiles must read u^n, so in EXP mode the source is a copy of u^n and in
// PHI mode the residual array (computed from u^n before this launch).
#include <algorithm>
#include <cstdlib>
#include <type_traits>

#include <cooperative_groups.h>

#include "gemv_acc.cuh"
#include "lem_internal.h"

namespace lem {

namespace {

// Four propagator rows per warp, 8 lanes per row: y_i = sum_k P[i, k] w[k]. With vec (row
// length a multiple of the vector width, rows 16-byte aligned) each lane streams its row in
// 16-byte loads, four in flight; else scalar loads. Several rows in flight per warp keep the
// load pipe busy through each row's reduction and owner update. A launch may be chained to the
// residual's: the blocks load their first chunks, then wait for it.
// What bounds it: HBM, and how many blocks are resident to keep loads in flight (hence 40 registers
// for FP32 rows); FP32 sums also took 60 % of the issue slots before they were packed; FP64 rows are
// near the FP64 pipe's rate. 320^2 variable diffusion (308 MB
// a step, its floor 45 us), a call of ten steps: 690 us; chained 674, the first 32 MB kept in L2 659,
// packed sums, windows staged without divisions and owner values read before their row 578, first
// chunks before the wait 564 to 573 (five blocks an SM 599, three chunks in flight 608). FP64 rows of
// the same problem 1499 -> 1456 us, 101^2 with tiles of 12 212 -> 169. A Schroedinger line of 65536
// (63 MB): 286, 270, 254, 206 us, its FP64 rows 822 -> 753.
// CPLX: complex states (interleaved re, im) with real-embedded propagators
// [[Re P, -Im P], [Im P, Re P]]: the window is staged as [re parts | im parts] (n_loc / 2 nodes
// each, zero padded); each owner's Re and Im rows are read once, left halves only.
constexpr int tiles_threads(int value, bool cplx) { return cplx && value == 4 ? 128 : 256; }
constexpr int tiles_blocks(int value, bool cplx) { return cplx ? (value == 4 ? 8 : 4) : (value == 4 ? 6 : 5); }
template <typename PT, bool CPLX>
__global__ void __launch_bounds__(tiles_threads(sizeof(PT), CPLX), tiles_blocks(sizeof(PT), CPLX))
    gemv_tiles_kernel(const PT* __restrict__ P, int64_t n_int, int64_t n_loc, const TileDesc* __restrict__ tiles,
                      const double* __restrict__ src, double* __restrict__ u, int64_t ny, int64_t nx, int accumulate,
                      int rsplit, int resident) {
  // the tile's window values, converted once to the propagator's precision
  extern __shared__ __align__(16) unsigned char wraw[];
  PT* w = reinterpret_cast<PT*>(wraw);
  // rsplit blocks share a tile, each taking a contiguous share of its owner rows: several
  // waves of short blocks instead of one wave of long ones (a shorter tail)
  const int t = blockIdx.x / rsplit, part = blockIdx.x % rsplit;
  const TileDesc td = tiles[t];
  const int wn = td.wext[0] * td.wext[1];  // window nodes
  const int hn = int(n_loc / 2);            // CPLX: padded window nodes
  const int wl = CPLX ? int(n_loc) : wn;    // staged window values
  const PT* Pt = P + int64_t(td.cls) * n_int * n_loc;
  const int ien = td.iext[0] * td.iext[1];  // owner nodes
  const int ie_all = ien;                   // owner nodes of this tile (CPLX: one group does both parts)
  const int rows_per = (ie_all + rsplit - 1) / rsplit;
  const int ib = part * rows_per, ie = min(ie_all, ib + rows_per);
  constexpr int V = 16 / sizeof(PT);
  const bool vec = (n_loc % V) == 0;  // (a row's end short of a whole chunk is masked, row_end)
  const unsigned long long policy = l2_policy(td.cls < resident);
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32, nw = blockDim.x / 32;
  const int grp = lane / 8, gl = lane % 8;
  // real rows: chunks j0 + gl + 8 k of a row; the first ones before the residual is waited for
  constexpr int U = 4;  // 16-byte loads in flight per lane
  const int nv = (wl + V - 1) / V;
  const bool ragged = wl % V != 0;
  int4 q[U];
  auto load = [&](int row, int j0) {
    const int4* r4 = reinterpret_cast<const int4*>(Pt + int64_t(row) * n_loc) + j0 + gl;
    if (j0 + 8 * U <= nv) {
#pragma unroll
      for (int k = 0; k < U; ++k) q[k] = load_policy(r4 + 8 * k, policy);
    } else {
#pragma unroll
      for (int k = 0; k < U; ++k) q[k] = j0 + 8 * k + gl < nv ? load_policy(r4 + 8 * k, policy) : make_int4(0, 0, 0, 0);
    }
  };
  if (!CPLX && vec && ib + warp * 4 < ie) load(min(ib + warp * 4 + grp, ie - 1), 0);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  // the window: node k = (a, b), then blockDim.x nodes further each time; zeros to a whole chunk
  const int wx = td.wext[1], step_a = int(blockDim.x) / wx, step_b = int(blockDim.x) % wx;
  for (int k = threadIdx.x, a = k / wx, b = k % wx; k < (CPLX ? hn : min((wn + V - 1) / V * V, int(n_loc)));
       k += blockDim.x, a += step_a, b += step_b) {
    if (b >= wx) {
      b -= wx;
      ++a;
    }
    if (k >= wn) {
      w[k] = PT(0);
      if (CPLX) w[hn + k] = PT(0);
      continue;
    }
    int64_t gy = int64_t(td.org[0]) + a, gx = int64_t(td.org[1]) + b;
    gy = gy < 0 ? gy + ny : (gy >= ny ? gy - ny : gy);
    gx = gx < 0 ? gx + nx : (gx >= nx ? gx - nx : gx);
    if (CPLX) {
      const double2 v = *reinterpret_cast<const double2*>(src + 2 * (gy * nx + gx));
      to_prec(v.x, w[k]);
      to_prec(v.y, w[hn + k]);
    } else {
      to_prec(src[gy * nx + gx], w[k]);
    }
  }
  __syncthreads();
  if constexpr (CPLX) {
    // complex: a row group per owner node o, reading its Re row (row o) and Im row (row
    // n_int / 2 + o) of the stored embedding, left halves only (the right halves repeat them):
    //   y_re = Re w_re - Im w_im,   y_im = Im w_re + Re w_im
    const int hl = hn;  // window columns per part
    const bool cvec = (n_loc % V) == 0 && (hl % V) == 0;
    for (int o0 = ib + warp * 4; o0 < ie; o0 += nw * 4) {
      const int o = o0 + grp;
      const bool live = o < ie;
      const int oc = live ? o : ib;  // (groups past the last row read a row of the share, and drop it)
      const PT* rre = Pt + int64_t(oc) * n_loc;
      const PT* rim = Pt + int64_t(int(n_int / 2) + oc) * n_loc;
      const int64_t p = int64_t(td.t0[0] + oc / td.iext[1]) * nx + td.t0[1] + oc % td.iext[1];
      double br = 0.0, bi = 0.0;  // (read before the row, whose time hides theirs)
      if (accumulate && gl == 0) {
        br = u[2 * p];
        bi = u[2 * p + 1];
      }
      typename std::conditional<sizeof(PT) == 8, AccCD, AccCF>::type acc;
      if (cvec) {
        // FP32 rows: four 16-byte loads per lane and row in flight, so a window of up to 128
        // nodes takes one round trip per row pair; FP64 rows are bound by the FP64 pipe.
        constexpr int CU = sizeof(PT) == 4 ? 4 : 2;
        const int nv = hl / V;
        const int4* a4 = reinterpret_cast<const int4*>(rre);
        const int4* b4 = reinterpret_cast<const int4*>(rim);
        for (int j = gl; j < nv; j += 8 * CU) {
          int4 qa[CU], qb[CU];
#pragma unroll
          for (int k = 0; k < CU; ++k) {
            const bool ok = j + 8 * k < nv;
            qa[k] = ok ? load_policy(a4 + j + 8 * k, policy) : make_int4(0, 0, 0, 0);
            qb[k] = ok ? load_policy(b4 + j + 8 * k, policy) : make_int4(0, 0, 0, 0);
          }
#pragma unroll
          for (int k = 0; k < CU; ++k) {
            if (j + 8 * k >= nv) break;
            const int4 wr4 = *reinterpret_cast<const int4*>(w + (j + 8 * k) * V);
            const int4 wi4 = *reinterpret_cast<const int4*>(w + hl + (j + 8 * k) * V);
            acc.chunk(reinterpret_cast<const PT*>(&qa[k]), reinterpret_cast<const PT*>(&qb[k]),
                      reinterpret_cast<const PT*>(&wr4), reinterpret_cast<const PT*>(&wi4));
          }
        }
      } else {
        for (int k = gl; k < hl; k += 8) acc.add(rre[k], rim[k], w[k], w[hl + k]);
      }
      double yr, yi;
      group_reduce(acc, yr, yi);
      if (live && gl == 0) {
        u[2 * p] = accumulate ? br + yr : yr;
        u[2 * p + 1] = accumulate ? bi + yi : yi;
      }
    }
  } else {
    // every lane runs the same number of row iterations (the shuffles need the whole warp)
    for (int i0 = ib + warp * 4; i0 < ie; i0 += nw * 4) {
      const int i = i0 + grp;
      const bool live = i < ie;
      const int ic = live ? i : ib;  // (groups past the last row read a row of the share, and drop it)
      const int64_t p = int64_t(td.t0[0] + ic / td.iext[1]) * nx + td.t0[1] + ic % td.iext[1];
      const double before = accumulate && gl == 0 ? u[p] : 0.0;  // (read before the row, whose time hides its)
      typename std::conditional<sizeof(PT) == 8, AccD, AccF>::type acc;
      if (vec) {
        const int4* w4 = reinterpret_cast<const int4*>(w);
        for (int j0 = 0;;) {
          if (j0 + 8 * U <= wl / V) {
#pragma unroll
            for (int k = 0; k < U; ++k) {
              const int4 wq = w4[j0 + 8 * k + gl];
              acc.chunk(reinterpret_cast<const PT*>(&q[k]), reinterpret_cast<const PT*>(&wq));
            }
          } else {
#pragma unroll
            for (int k = 0; k < U; ++k) {
              const int j = j0 + 8 * k + gl;
              if (j >= nv) break;
              const int4 wq = w4[j];
              if (ragged) row_end(q[k], Pt, wl - j * V);
              acc.chunk(reinterpret_cast<const PT*>(&q[k]), reinterpret_cast<const PT*>(&wq));
            }
          }
          if ((j0 += 8 * U) >= nv) break;
          load(ic, j0);
        }
        if (i0 + nw * 4 < ie) load(min(i + nw * 4, ie - 1), 0);
      } else {
        const PT* row = Pt + int64_t(ic) * n_loc;
        for (int k = gl; k < wl; k += 8) acc.add(row[k], w[k]);
      }
      const double y = group_reduce(acc);
      if (live && gl == 0) u[p] = accumulate ? before + y : y;
    }
  }
}

// The defect of the third-order Rosenbrock step, times two: 2 dt (G(U) - G(u)) with
// G(v) = F(v) - J(u_m) v. The linear parts cancel, so it is pointwise:
// 2 dt [(U - U^3) - (u - u^3) - (1 - 3 u_m^2)(U - u)].
__global__ void rb3_defect_kernel(const double* __restrict__ U, const double* __restrict__ u,
                                  const double* __restrict__ um, double dt, double* __restrict__ d, int64_t n) {
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
    const double Ui = U[i], ui = u[i], mi = um[i];
    d[i] = 2.0 * dt * ((Ui - Ui * Ui * Ui) - (ui - ui * ui * ui) - (1.0 - 3.0 * mi * mi) * (Ui - ui));
  }
}

__global__ void f64_to_f32_kernel(const double* __restrict__ a, float* __restrict__ b, int64_t n) {
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x)
    b[i] = __double2float_rn(a[i]);
}

}  // namespace


// FP32 copy of the propagators for the reduced-precision GEMV (refreshed after each build).
lem_status gemv_prepare_f32(lem_ctx* ctx) {
  const int64_t n = int64_t(ctx->classes.size()) * ctx->n_int * ctx->n_loc;
  if (!ctx->d_P32) LEM_TRY(dev_alloc(ctx, reinterpret_cast<void**>(&ctx->d_P32), sizeof(float) * n));
  f64_to_f32_kernel<<<1024, 256, 0, ctx->stream>>>(ctx->d_P, ctx->d_P32, n);
  if (ctx->d_P3) {
    if (!ctx->d_P3_32) LEM_TRY(dev_alloc(ctx, reinterpret_cast<void**>(&ctx->d_P3_32), sizeof(float) * n));
    f64_to_f32_kernel<<<1024, 256, 0, ctx->stream>>>(ctx->d_P3, ctx->d_P3_32, n);
  }
  LEM_CUDA_TRY(cudaGetLastError());
  ctx->p32_gen = ctx->build_gen;
  return LEM_OK;
}

// ---------------------------------------------------------------- persistent multi-step
// Small problems (config 1: 16 tiles of a 1024-node mesh) are bound by launch latency, two
// launches per step. This cooperative kernel runs all nsteps in one launch. Per step every
// block takes its tiles: it forms the window's source straight from u^n (the residual dt A u^n
// at each window node in PHI mode, u^n in EXP mode) in shared memory, applies the tile's
// propagator (four rows per warp) and writes the owner values of u^{n+1} into the other state
// buffer; one grid barrier ends the step. Linear real problems on the GEMV path only (no
// Jacobian refresh, one scheme stage).
// A tile's owner rows are shared out over rsplit blocks (each stages the tile's window), so that a
// handful of tiles still uses the device: the FP64 pipe does 2 multiply-adds per clock and SM, and
// one block per tile of 64 x 96 took most of a step (16 tiles: 5.6 us a step).
// SMEMP: one share of a tile per block, its propagator rows kept in shared memory for all steps.
static int persist_threads(int rsplit) { return rsplit > 1 ? 128 : 256; }
// BLOCKS: how many an SM holds at least (its registers). Four leave the FP32 rows what they want; five
// where the tiles then take a round less: a line of 120 000 nodes (1875 tiles), ten steps 272 us in four
// rounds, 228 in three; 60 000 nodes (two rounds either way) 138 and 146.
template <typename PT, bool SMEMP, int BLOCKS>
__global__ void __launch_bounds__(256, BLOCKS) gemv_persistent_kernel(const PT* __restrict__ P, int64_t n_int, int64_t n_loc,
                                                              const TileDesc* __restrict__ tiles, int ntiles,
                                                              const double* __restrict__ coef, int64_t cstride,
                                                              int64_t ny, int64_t nx, int ndim, int pery, int perx,
                                                              int phi, double* __restrict__ src,
                                                              double* __restrict__ u, int nsteps, int rsplit) {
  namespace cg = cooperative_groups;
  cg::grid_group grid = cg::this_grid();
  extern __shared__ __align__(16) unsigned char wraw[];
  PT* w = reinterpret_cast<PT*>(wraw);
  const int64_t npts = ny * nx;
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32, nw = blockDim.x / 32;
  const int grp = lane / 8, gl = lane % 8;
  using Acc = typename std::conditional<sizeof(PT) == 8, AccD, AccF>::type;
  // SMEMP: the block's tile propagator (n_int x n_loc) after the window buffer
  PT* Ps = reinterpret_cast<PT*>(wraw + ((sizeof(double) * size_t(n_loc) + 15) & ~size_t(15)));
  // owner rows [*ib, *ie) of share `part` of a tile (shares are whole groups of 4 rows)
  auto share = [&](const TileDesc& td, int part, int* ib, int* ie) {
    const int owners = td.iext[0] * td.iext[1];
    const int per = rsplit == 1 ? owners : ((owners + rsplit - 1) / rsplit + 3) / 4 * 4;
    *ib = min(owners, part * per);
    *ie = min(owners, *ib + per);
  };
  if (SMEMP) {
    const TileDesc td = tiles[rsplit == 1 ? blockIdx.x : blockIdx.x / rsplit];
    int ib, ie;
    share(td, rsplit == 1 ? 0 : blockIdx.x % rsplit, &ib, &ie);
    const PT* src_p = P + (int64_t(td.cls) * n_int + ib) * n_loc;
    for (int64_t e = threadIdx.x; e < (ie - ib) * n_loc; e += blockDim.x) Ps[e] = src_p[e];
    __syncthreads();
  }
  // u^n and u^{n+1} alternate between u and src (every node has exactly one owner tile, so
  // each step writes the whole of the other buffer); one grid barrier per step
  double* cur = u;
  double* nxt = src;
  for (int step = 0; step < nsteps; ++step) {
    for (int t = blockIdx.x; t < ntiles * rsplit; t += gridDim.x) {
      const TileDesc td = tiles[rsplit == 1 ? t : t / rsplit];
      const int wl = td.wext[0] * td.wext[1];
      int ib, ie;
      share(td, rsplit == 1 ? 0 : t % rsplit, &ib, &ie);
      // the window's source from u^n: the residual dt A u^n at each window node (PHI), or u^n
      for (int k = threadIdx.x; k < wl; k += blockDim.x) {
        const int a = td.wext[0] == 1 ? 0 : k / td.wext[1], b = k - a * td.wext[1];
        int64_t gy = int64_t(td.org[0]) + a, gx = int64_t(td.org[1]) + b;
        gy = gy < 0 ? gy + ny : (gy >= ny ? gy - ny : gy);
        gx = gx < 0 ? gx + nx : (gx >= nx ? gx - nx : gx);
        const int64_t p = gy * nx + gx;
        double v = cur[p];
        if (phi) {
          auto cf = [&](int c) { return cstride ? coef[int64_t(c) * npts + p] : coef[c]; };
          double acc = cf(0) * v;
          if (gx > 0) acc = fma(cf(1), cur[p - 1], acc);
          else if (perx) acc = fma(cf(1), cur[p + nx - 1], acc);
          if (gx + 1 < nx) acc = fma(cf(2), cur[p + 1], acc);
          else if (perx) acc = fma(cf(2), cur[p + 1 - nx], acc);
          if (ndim == 2) {
            if (gy > 0) acc = fma(cf(3), cur[p - nx], acc);
            else if (pery) acc = fma(cf(3), cur[p + (ny - 1) * nx], acc);
            if (gy + 1 < ny) acc = fma(cf(4), cur[p + nx], acc);
            else if (pery) acc = fma(cf(4), cur[p - (ny - 1) * nx], acc);
          }
          v = acc;
        }
        w[k] = PT(v);
      }
      if (threadIdx.x < 4 && wl + threadIdx.x < n_loc) w[wl + threadIdx.x] = PT(0);  // to a whole chunk
      __syncthreads();
      const PT* Pt = SMEMP ? Ps - int64_t(ib) * n_loc : P + int64_t(td.cls) * n_int * n_loc;
      constexpr int V = 16 / sizeof(PT);
      const bool vec = (n_loc % V) == 0;
      for (int i0 = ib + warp * 4; i0 < ie; i0 += nw * 4) {
        const int i = i0 + grp;
        const bool live = i < ie;
        const PT* row = Pt + int64_t(live ? i : ib) * n_loc;
        // the same partition of a row over the 8 lanes, and the same order, as gemv_tiles_kernel
        // (16-byte chunks j = lane, lane + 8, ... when rows allow them): bit-identical results
        Acc acc;
        if (live) {
          if (vec) {
            const int4* r4 = reinterpret_cast<const int4*>(row);
            for (int j = gl; j < (wl + V - 1) / V; j += 8) {
              int4 q = SMEMP ? r4[j] : __ldcs(r4 + j);
              if (wl % V != 0) row_end(q, row, wl - j * V);
              acc.chunk(reinterpret_cast<const PT*>(&q), w + j * V);
            }
          } else {
            for (int k = gl; k < wl; k += 8) acc.add(row[k], w[k]);
          }
        }
        const double y = group_reduce(acc);
        if (live && gl == 0) {
          const int64_t p = int64_t(td.t0[0] + i / td.iext[1]) * nx + td.t0[1] + i % td.iext[1];
          nxt[p] = phi ? cur[p] + y : y;
        }
      }
      __syncthreads();  // the window buffer is reused by the block's next tile
    }
    grid.sync();  // u^{n+1} complete before any block reads it
    double* tmp = cur;
    cur = nxt;
    nxt = tmp;
  }
  if (cur != u)  // an odd number of steps ended in the scratch buffer
    for (int64_t p = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; p < npts; p += int64_t(gridDim.x) * blockDim.x)
      u[p] = cur[p];
}

// Whether lem_step may run its steps in one persistent launch, and with how many blocks; *rsplit:
// blocks per tile (at most one block per SM then, of 8 rows at least), *fn: the kernel.
static int persistent_blocks(lem_ctx* ctx, bool f32, int nsteps, int* rsplit, const void** fn) {
  *rsplit = 1;
  const lem_problem_desc& d = ctx->desc;
  if (nsteps < 2 || d.reaction || d.scheme != LEM_SCHEME_EULER || ctx->cplx) return 0;
  if (ctx->npts > (int64_t(1) << 20) || ctx->tiles.size() > 4096) return 0;
  if (std::getenv("LEM_NO_PERSISTENT")) return 0;  // switch for comparisons
  int dev_coop = 0, nsm = 0, per_sm = 0;
  if (cudaDeviceGetAttribute(&dev_coop, cudaDevAttrCooperativeLaunch, ctx->device) != cudaSuccess || !dev_coop ||
      cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, ctx->device) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  const size_t smem = sizeof(double) * size_t(ctx->n_loc);
  // one block per share of a tile, within what the device holds at once
  const int64_t nt = int64_t(ctx->tiles.size());
  *rsplit = int(std::max<int64_t>(1, std::min<int64_t>(nsm / nt, ctx->n_int / 8)));
  const int threads = persist_threads(*rsplit);
  auto rounds = [&](const void* fn) {  // of the device, over the tiles; 0: not even one block an SM
    per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, threads, smem) != cudaSuccess || per_sm < 1) {
      cudaGetLastError();
      return int64_t(0);
    }
    return (nt * *rsplit + int64_t(per_sm) * nsm - 1) / (int64_t(per_sm) * nsm);
  };
  *fn = f32 ? reinterpret_cast<const void*>(gemv_persistent_kernel<float, false, 4>)
            : reinterpret_cast<const void*>(gemv_persistent_kernel<double, false, 4>);
  const int64_t r4 = rounds(*fn);
  if (r4 == 0) return 0;
  if (f32 && r4 > 1) {
    const int four = per_sm;
    const void* five = reinterpret_cast<const void*>(gemv_persistent_kernel<float, false, 5>);
    const int64_t r5 = rounds(five);
    if (r5 > 0 && r5 < r4) *fn = five;
    else per_sm = four;
  }
  return int(std::min<int64_t>(int64_t(per_sm) * nsm, nt * *rsplit));
}

lem_status step_gemv_multi(lem_ctx* ctx, double* d_u, int nsteps, bool f32, bool* done) {
  *done = false;
  int rsplit = 1;
  const void* fn = nullptr;
  const int blocks = persistent_blocks(ctx, f32, nsteps, &rsplit, &fn);
  if (blocks < 1) return LEM_OK;
  if (f32 && ctx->p32_gen != ctx->build_gen) LEM_TRY(gemv_prepare_f32(ctx));
  const lem_problem_desc& d = ctx->desc;
  // one share per block with propagator rows few enough for shared memory: keep them there
  const size_t wbytes = (sizeof(double) * size_t(ctx->n_loc) + 15) & ~size_t(15);
  const size_t rows = size_t((ctx->n_int + rsplit - 1) / rsplit + 3) / 4 * 4;
  const size_t pbytes = (f32 ? sizeof(float) : sizeof(double)) * rows * size_t(ctx->n_loc);
  bool smemp = int64_t(blocks) == int64_t(ctx->tiles.size()) * rsplit && wbytes + pbytes <= 200 * 1024 &&
               std::getenv("LEM_NO_SMEM_P") == nullptr;
  const void* fn_s = f32 ? reinterpret_cast<const void*>(gemv_persistent_kernel<float, true, 4>)
                         : reinterpret_cast<const void*>(gemv_persistent_kernel<double, true, 4>);
  if (smemp) {  // every block must still be co-resident with the larger footprint
    int per_sm = 0, nsm = 0;
    if (allow_smem(fn_s, ctx->device, wbytes + pbytes) != cudaSuccess ||
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, ctx->device) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn_s, persist_threads(rsplit), wbytes + pbytes) != cudaSuccess ||
        int64_t(per_sm) * nsm < blocks) {
      cudaGetLastError();
      smemp = false;
    }
  }
  const size_t smem = smemp ? wbytes + pbytes : sizeof(double) * size_t(ctx->n_loc);
  if (smemp) fn = fn_s;
  int ntiles = int(ctx->tiles.size()), ndim = d.ndim, pery = ctx->bcy == LEM_BC_PERIODIC,
      perx = ctx->bcx == LEM_BC_PERIODIC, phi = d.mode == LEM_MODE_PHI;
  int64_t n_int = ctx->n_int, n_loc = ctx->n_loc, cstride = d.coef_stride, ny = ctx->ny, nx = ctx->nx;
  const void* P = f32 ? static_cast<const void*>(ctx->d_P32) : static_cast<const void*>(ctx->d_P);
  void* args[] = {&P, &n_int, &n_loc, &ctx->d_tiles, &ntiles, &ctx->d_coef, &cstride, &ny, &nx,
                  &ndim, &pery, &perx, &phi, &ctx->d_r, &d_u, &nsteps, &rsplit};
  cudaEvent_t stop;
  LEM_CUDA_TRY(ctx->timing_begin(&stop));
  LEM_CUDA_TRY(cudaLaunchCooperativeKernel(fn, dim3(blocks), dim3(persist_threads(rsplit)), args, smem, ctx->stream));
  ctx->timing_end(stop);
  *done = true;
  return LEM_OK;
}

// Threads per GEMV block: 128 for the complex FP32 kernel (short rows, little work per block,
// more blocks resident per SM), 256 otherwise.
static int gemv_threads(const lem_ctx* ctx, bool f32) { return tiles_threads(f32 ? 4 : 8, ctx->cplx); }

// Blocks per tile: about four waves of blocks (6 to 8 resident per SM), at least 32 owner rows
// per block, each block's share a whole number of passes (a pass: 4 rows per warp), so that no
// pass runs part empty (512^2 variable diffusion: 4 blocks of 64 rows per tile, not 5 of 52).
int gemv_row_split(const lem_ctx* ctx, int threads) {
  const int64_t nt = int64_t(ctx->tiles.size());
  int nsm = 0;
  if (cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, ctx->device) != cudaSuccess || nsm < 1) nsm = 152;
  const int rmax = std::max<int>(1, int(ctx->n_int / 32));
  int rsplit = std::max(1, std::min<int>(rmax, int((4LL * 8 * nsm + nt - 1) / nt)));
  const int owners = int(ctx->cplx ? ctx->n_int / 2 : ctx->n_int), pass = threads / 8;
  const int rows = ((owners + rsplit - 1) / rsplit + pass - 1) / pass * pass;
  return std::max(1, (owners + rows - 1) / rows);
}

// Classes whose propagators are to stay in L2 from step to step: the first 32 MB (129 MB of L2 serve two
// dies, and hold the state, the coefficients and what passes through as well). All others are read
// as passing through. A call of ten steps on 320^2 variable diffusion (308 MB a step): 32 MB 571.6 us,
// 48 MB 572.5, 80 MB 586 (before sums were packed: none 674, 32 MB 659); a Schroedinger line of 65536
// (63 MB, 416 of 820 classes kept): 206 us, with room for all of it 218 (before: none 270, kept 254).
static int resident_classes(const lem_ctx* ctx, bool f32) {
  const int64_t bytes = ctx->n_int * ctx->n_loc * (f32 ? 4 : 8) / (ctx->cplx ? 2 : 1);
  return int(std::min<int64_t>(32000000 / std::max<int64_t>(bytes, 1), int64_t(ctx->classes.size())));
}

// Shared memory a block for a chained launch of FP64 rows that fills less than a wave. Its blocks are
// placed while the residual's still run, on whatever SM has room, and the SMs with most of them set the time
// (the FP64 pipe's): no more of them fit an SM than an even spread puts there. 112^2 variable
// diffusion, tiles of 16 (392 blocks), ten steps: 330 us placed anyhow, 293 without the chain, 254 so;
// 128^2 (512 blocks) 386, 355, 339.
static size_t spread_smem(unsigned blocks, int resident, size_t smem, int device) {
  int nsm = 0, room = 0;
  if (cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, device) != cudaSuccess || nsm < 1 ||
      cudaDeviceGetAttribute(&room, cudaDevAttrMaxSharedMemoryPerMultiprocessor, device) != cudaSuccess) {
    cudaGetLastError();
    return smem;
  }
  const int per = int((blocks + nsm - 1) / nsm);
  if (per >= resident) return smem;
  const size_t even = size_t(room / per - 1024) / 128 * 128 - 128;  // (1 KB a block is the system's)
  return std::max(smem, even);
}

// One LEM step by the batched GEMV: PHI reads the residual, EXP a copy of u^n.
lem_status step_gemv(lem_ctx* ctx, double* d_u, bool f32) {
  cudaStream_t st = ctx->stream;
  const bool phi = ctx->desc.mode == LEM_MODE_PHI;
  const bool rb3 = ctx->desc.scheme == LEM_SCHEME_RB3 && ctx->desc.reaction;  // (linear: the defect is 0)
  // (before the residual: the streamed apply reads propagators while the residual still runs)
  if (f32 && ctx->p32_gen != ctx->build_gen) LEM_TRY(gemv_prepare_f32(ctx));
  if (rb3)
    LEM_CUDA_TRY(cudaMemcpyAsync(ctx->d_u0, d_u, sizeof(double) * ctx->npts, cudaMemcpyDeviceToDevice, st));
  const double* src;
  if (phi) {
    LEM_CUDA_TRY(launch_residual_fp64(ctx, ctx->d_r, d_u));
    src = ctx->d_r;
  } else {
    LEM_CUDA_TRY(cudaMemcpyAsync(ctx->d_r, d_u, sizeof(double) * ctx->npts * (ctx->cplx ? 2 : 1),
                                 cudaMemcpyDeviceToDevice, st));
    src = ctx->d_r;
  }
  const size_t smem = sizeof(double) * size_t(ctx->n_loc);
  const unsigned nt = unsigned(ctx->tiles.size());
  const int threads = gemv_threads(ctx, f32);
  const int rsplit = gemv_row_split(ctx, threads);
  cudaEvent_t stop;
  LEM_CUDA_TRY(ctx->timing_begin(&stop));
  auto gemv = [&](const double* P64, const float* P32, const double* x, bool after_residual) -> lem_status {
    const int acc = phi ? 1 : 0;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(nt * rsplit);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = f32 || ctx->cplx ? smem : spread_smem(nt * rsplit, tiles_blocks(8, false), smem, ctx->device);
    cfg.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = after_residual ? 1 : 0;  // (it waits for the residual before the windows only)
    auto go = [&](auto kernel, auto P) -> lem_status {
      LEM_CUDA_TRY(cudaLaunchKernelEx(&cfg, kernel, P, ctx->n_int, ctx->n_loc,
                                      static_cast<const TileDesc*>(ctx->d_tiles), x, d_u, ctx->ny, ctx->nx,
                                      acc, rsplit, resident_classes(ctx, f32)));
      return LEM_OK;
    };
    if (f32) return ctx->cplx ? go(gemv_tiles_kernel<float, true>, P32) : go(gemv_tiles_kernel<float, false>, P32);
    return ctx->cplx ? go(gemv_tiles_kernel<double, true>, P64) : go(gemv_tiles_kernel<double, false>, P64);
  };
  LEM_TRY(gemv(ctx->d_P, ctx->d_P32, src, phi));
  if (rb3) {  // second stage: u^{n+1} = U + 2 phi_3(dt J_m) dt (G(U) - G(u^n)), window by window
    rb3_defect_kernel<<<1024, 256, 0, st>>>(d_u, ctx->d_u0, ctx->d_um, ctx->desc.dt, ctx->d_r, ctx->npts);
    LEM_TRY(gemv(ctx->d_P3, ctx->d_P3_32, ctx->d_r, false));
  }
  ctx->timing_end(stop);
  LEM_CUDA_TRY(cudaGetLastError());
  return LEM_OK;
}

// One FP64 GEMV step of a real exponential-Euler problem with caller-provided scratch r (npts
// doubles): the kernels and launch shape of step_gemv, so the result is the same bit for bit.
// Used by the allocation-free entry point.
lem_status step_gemv_scratch(lem_ctx* ctx, double* d_u, double* r) {
  cudaStream_t st = ctx->stream;
  if (ctx->desc.mode == LEM_MODE_PHI) {
    LEM_CUDA_TRY(launch_residual_fp64(ctx, r, d_u));
  } else {
    LEM_CUDA_TRY(cudaMemcpyAsync(r, d_u, sizeof(double) * ctx->npts, cudaMemcpyDeviceToDevice, st));
  }
  const size_t smem = sizeof(double) * size_t(ctx->n_loc);
  const unsigned nt = unsigned(ctx->tiles.size());
  const int threads = gemv_threads(ctx, false);
  const int rsplit = gemv_row_split(ctx, threads);
  const int acc = ctx->desc.mode == LEM_MODE_PHI ? 1 : 0;
  gemv_tiles_kernel<double, false><<<nt * rsplit, threads, smem, st>>>(ctx->d_P, ctx->n_int, ctx->n_loc, ctx->d_tiles,
                                                                       r, d_u, ctx->ny, ctx->nx, acc, rsplit,
                                                                       resident_classes(ctx, false));
  LEM_CUDA_TRY(cudaGetLastError());
  return LEM_OK;
}

lem_status gemv_set_smem(lem_ctx* ctx) {
  const size_t bytes = sizeof(double) * size_t(ctx->n_loc);
  LEM_CUDA_TRY(allow_smem(reinterpret_cast<const void*>(gemv_tiles_kernel<double, false>), ctx->device, 0));  // (spread_smem)
  if (bytes > 48 * 1024)
    for (const void* k : {reinterpret_cast<const void*>(gemv_tiles_kernel<float, false>),
                          reinterpret_cast<const void*>(gemv_tiles_kernel<double, false>),
                          reinterpret_cast<const void*>(gemv_tiles_kernel<float, true>),
                          reinterpret_cast<const void*>(gemv_tiles_kernel<double, true>)})
      LEM_CUDA_TRY(allow_smem(k, ctx->device, bytes));
  return LEM_OK;
}

}  // namespace lem
