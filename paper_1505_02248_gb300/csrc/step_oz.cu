// FP64 LEM step on the tensor cores (Sec. 3 steps 1-3, Eq. lem), for contexts whose tiles share
// propagators: exact digit products (oz_core.cuh) in place of FP64 multiply-adds.
//
//   PHI:  r = dt F(u^n); the windows of r, cut into digits (gather and cut in one pass);
//         y = P r|_M for 128 windows x 64 owner rows per CTA; u_D += y.
//   EXP:  the windows of u^n, cut; u_D = P u|_M.
//
// GB300's FP64 pipe runs 1.1 TFLOP/s, its FP16 tensor cores 1900. The 1024^2 periodic problem
// (1024 windows of 2304 nodes, 1024 x 2304 propagator) took 4.67 ms a step as one FP64 GEMM, at
// the FP64 pipe's rate, and takes 0.145 ms here (products 113 us, window digits 20, residual 15); a
// walled 389 x 517 mesh with 16 classes, their GEMMs one after another, 29.2 ms a step, and 0.112
// ms here.
//
// Layout: windows are the rows of A (128 windows of one class form a block), owner rows of the
// class's propagator the columns of B. The propagators are cut once per build. One launch covers
// every class: a unit is (window block, 64 owner rows), so classes with few windows (walls,
// corners) run beside the large ones instead of after them.
//
// Split over K: when the units leave SMs idle, the K blocks of a unit are divided over a cluster
// of 2, 4 or 8 CTAs; each then sums the others' 64-bit level sums over distributed shared memory
// for its share of the columns. Integer sums: the result does not depend on the split.
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>
#include <new>
#include <string>
#include <vector>

#include "lem_internal.h"
#include "oz_core.cuh"

namespace lem {

namespace {

namespace cg = cooperative_groups;

struct WinBlock {   // up to 128 windows of one class
  int32_t first;    // first entry in class_order
  int32_t count;
  int32_t cls;
  int32_t nkb;      // K blocks of 16 window nodes
  int64_t a_off;    // halves into the window digits
  int32_t e_off;    // scale exponents of its rows
  int32_t pad;
};
struct Unit {
  int32_t wb;       // window block
  int32_t col0;     // first owner row
  int32_t ncol;     // owner rows of the class from col0 on (may exceed 64)
  int32_t f_off;    // scale exponents of the owner rows
  int64_t b_off;    // halves into the propagator digits
};
struct PropRows {   // 64 owner rows of one class
  int32_t cls, row0, rows, cols, nkb, f_off;
  int64_t b_off;
};

// k / d for 0 <= k < 2^16 and 1 < d < 2^16 by one multiply (inv = div_inv(d)); d = 1: inv = 0.
__host__ __device__ __forceinline__ uint32_t div_inv(uint32_t d) { return d > 1 ? 0xFFFFFFFFu / d + 1u : 0u; }
__device__ __forceinline__ int div_by(int k, uint32_t inv) { return inv ? int(__umulhi(uint32_t(k), inv)) : k; }

// Window digits: a CTA cuts R windows of one block (8: one core-matrix row group, so the 16-byte
// stores of 8 lanes fill 128 bytes; fewer where 8 a CTA would leave SMs idle). Its warps find each
// window's largest exponent, then each thread cuts 8 consecutive nodes of one window. Bound by
// the 14 bytes written per node and about 40 integer operations; the two reads of the window come
// from L2. (Eight windows per 256-thread CTA and 64-bit node arithmetic: 43 us for 1024 windows
// of 2304 nodes.)
constexpr int WIN_THREADS = 512;
template <int R>
__global__ void __launch_bounds__(WIN_THREADS) oz_windows_kernel(const double* __restrict__ src,
                                                                 const TileDesc* __restrict__ tiles,
                                                                 const int32_t* __restrict__ order,
                                                                 const WinBlock* __restrict__ blocks, int wb0, int ny,
                                                                 int nx, int* __restrict__ e, __half* __restrict__ out) {
  constexpr int PER = oz::BM / R;  // CTAs per block
  const WinBlock b = blocks[wb0 + blockIdx.x / PER];
  const int r0 = (blockIdx.x % PER) * R;
  if (r0 >= b.count) return;
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  __shared__ int2 org[R];
  __shared__ int ex[R], wext[2];
  if (threadIdx.x < R) {
    const TileDesc& t = tiles[order[b.first + min(r0 + int(threadIdx.x), b.count - 1)]];
    org[threadIdx.x] = make_int2(t.org[0], t.org[1]);
    ex[threadIdx.x] = 0;
    if (threadIdx.x == 0) {  // one class: one window shape
      wext[0] = t.wext[0];
      wext[1] = t.wext[1];
    }
  }
  __syncthreads();
  const int wx = wext[1], wn = wext[0] * wx;
  const uint32_t inv = div_inv(uint32_t(wx));
  auto at = [&](int2 o, int a, int c) {  // (meshes hold at most 2^31 nodes)
    int gy = o.x + a, gx = o.y + c;
    gy = gy < 0 ? gy + ny : (gy >= ny ? gy - ny : gy);
    gx = gx < 0 ? gx + nx : (gx >= nx ? gx - nx : gx);
    return src[uint32_t(gy) * uint32_t(nx) + uint32_t(gx)];
  };
  {
    constexpr int WPR = WIN_THREADS / 32 / R;  // warps per window
    const int r = warp / WPR;
    const int2 o = org[r];
    int E = 0;
#pragma unroll 4
    for (int k = (warp % WPR) * 32 + lane; k < wn; k += 32 * WPR) {
      const int a = div_by(k, inv);
      E = max(E, oz::exp_field(static_cast<unsigned long long>(__double_as_longlong(at(o, a, k - a * wx)))));
    }
    for (int q = 16; q > 0; q >>= 1) E = max(E, __shfl_xor_sync(0xffffffffu, E, q));
    if (lane == 0) atomicMax(&ex[r], E);
  }
  __syncthreads();
  const int r = threadIdx.x % R;
  const int sc = oz::scale_exp(ex[r]);
  if (threadIdx.x < R) e[b.e_off + r0 + r] = sc;
  const int er = sc == oz::kNonFinite ? 4096 : sc;  // (non-finite: every digit 0)
  const int2 o = org[r];
  __half* dst0 = out + b.a_off;
  for (int k8 = (threadIdx.x / R) * 8; k8 < b.nkb * oz::KB; k8 += WIN_THREADS / R * 8) {
    unsigned long long N[8];
    int a = div_by(k8, inv), c = k8 - a * wx;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const double v = k8 + u < wn ? at(o, a, c) : 0.0;
      N[u] = oz::biased_digits(static_cast<unsigned long long>(__double_as_longlong(v)), er);
      if (++c >= wx) {
        c = 0;
        ++a;
      }
    }
    oz::store_digits(dst0 + size_t(k8 / oz::KB) * oz::A_BLOCK + oz::tile_off(r0 + r, k8 % oz::KB), oz::A_SLICE, N);
  }
}

// Propagator digits, once per build: a CTA cuts 8 owner rows.
__global__ void __launch_bounds__(256) oz_prop_kernel(const double* __restrict__ P, int64_t n_int, int64_t n_loc,
                                                      const PropRows* __restrict__ rows, int* __restrict__ f,
                                                      __half* __restrict__ out) {
  const PropRows p = rows[blockIdx.x / 8];
  const int r0 = (blockIdx.x % 8) * 8;
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  __shared__ int ex[8];
  auto row = [&](int i) { return P + (int64_t(p.cls) * n_int + p.row0 + i) * n_loc; };
  {
    int E = 0;
    if (r0 + warp < p.rows)
      for (int k = lane; k < p.cols; k += 32)
        E = max(E, oz::exp_field(static_cast<unsigned long long>(__double_as_longlong(row(r0 + warp)[k]))));
    for (int o = 16; o > 0; o >>= 1) E = max(E, __shfl_xor_sync(0xffffffffu, E, o));
    if (lane == 0) {
      ex[warp] = oz::scale_exp(E);
      f[p.f_off + r0 + warp] = ex[warp];
    }
  }
  __syncthreads();
  const int r = threadIdx.x % 8;
  const bool live = r0 + r < p.rows;
  const int er = ex[r] == oz::kNonFinite ? 4096 : ex[r];
  for (int k8 = (threadIdx.x / 8) * 8; k8 < p.nkb * oz::KB; k8 += 256) {
    unsigned long long N[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const double v = live && k8 + u < p.cols ? row(r0 + r)[k8 + u] : 0.0;
      N[u] = oz::biased_digits(static_cast<unsigned long long>(__double_as_longlong(v)), er);
    }
    oz::store_digits(out + p.b_off + size_t(k8 / oz::KB) * oz::B_BLOCK + oz::tile_off(r0 + r, k8 % oz::KB),
                     oz::B_SLICE, N);
  }
}

struct StepParams {
  const WinBlock* blocks;
  const Unit* units;
  const TileDesc* tiles;
  const int32_t* order;
  const __half* a;
  const __half* b;
  const int* e;
  const int* f;
  const double* P;     // (rows with infinities or NaN are formed in FP64)
  const double* src;
  double* u;
  int64_t n_int, n_loc, ny, nx;
  int unit0, ks, accumulate;
  int* err;
};

// The element of window `t` and owner row i in FP64, where an operand is not finite.
__device__ __noinline__ double plain_dot(const StepParams& p, const TileDesc& t, int i) {
  const double* row = p.P + (int64_t(t.cls) * p.n_int + i) * p.n_loc;
  const int wn = t.wext[0] * t.wext[1];
  double s = 0.0;
  for (int k = 0; k < wn; ++k) {
    int64_t gy = int64_t(t.org[0]) + k / t.wext[1], gx = int64_t(t.org[1]) + k % t.wext[1];
    gy = gy < 0 ? gy + p.ny : (gy >= p.ny ? gy - p.ny : gy);
    gx = gx < 0 ? gx + p.nx : (gx >= p.nx ? gx - p.nx : gx);
    s = fma(row[k], p.src[gy * p.nx + gx], s);
  }
  return s;
}

// One unit per cluster of ks CTAs (ks = 1: no cluster). The scatter adds each owner's increment
// to the state (PHI) or stores it (EXP); thread = column first, so a row's owners are written in
// runs of the tile width.
__global__ void __launch_bounds__(oz::THREADS, 1) oz_step_kernel(const __grid_constant__ StepParams p) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  __shared__ volatile int s_abort;
  const oz::Shared sh = oz::carve(smem_raw);
  const int ks = p.ks, rank = int(blockIdx.x) % ks;
  const Unit un = p.units[p.unit0 + int(blockIdx.x) / ks];
  const WinBlock wb = p.blocks[un.wb];
  __shared__ int64_t s_node[oz::BM];  // first owner node and scale exponent of each window
  __shared__ int s_e[oz::BM], s_f[oz::BN], s_ix;
  if (threadIdx.x < wb.count) {
    const TileDesc& t = p.tiles[p.order[wb.first + threadIdx.x]];
    s_node[threadIdx.x] = int64_t(t.t0[0]) * p.nx + t.t0[1];
    s_e[threadIdx.x] = p.e[wb.e_off + threadIdx.x];
    if (threadIdx.x == 0) s_ix = t.iext[1];
  } else if (threadIdx.x >= oz::BM && threadIdx.x < oz::BM + oz::BN) {
    s_f[threadIdx.x - oz::BM] = p.f[un.f_off + int(threadIdx.x) - oz::BM];
  }
  const uint32_t tmem = oz::setup(sh, &s_abort);
  const int k0 = wb.nkb * rank / ks, k1 = wb.nkb * (rank + 1) / ks;
  const bool any = k1 > k0;
  if (any)
    oz::products(sh, tmem, p.a + wb.a_off + size_t(k0) * oz::A_BLOCK, p.b + un.b_off + size_t(k0) * oz::B_BLOCK,
                 k1 - k0, p.err, &s_abort);
  longlong2* sums = reinterpret_cast<longlong2*>(sh.stage);
  cg::cluster_group cl = cg::this_cluster();
  if (ks > 1) {
    if (!any)
      for (int q = threadIdx.x; q < oz::BN * oz::SUM_PITCH; q += blockDim.x) sums[q] = make_longlong2(0, 0);
    cl.sync();
  }
  const int lcw = 6 - (31 - __clz(ks)), cw = 1 << lcw, c0 = rank * cw;  // this CTA's columns
  if (!s_abort && c0 < un.ncol) {
    const int ix = s_ix;
    const uint32_t inv = div_inv(uint32_t(ix));
    constexpr int U = 8;  // elements per thread in flight (the state is read before any is written)
    const int total = wb.count * cw;
    for (int q0 = threadIdx.x; q0 < total; q0 += U * oz::THREADS) {
      int64_t node[U];
      double old[U];
#pragma unroll
      for (int k = 0; k < U; ++k) {
        const int q = q0 + k * oz::THREADS, col = c0 + (q & (cw - 1)), row = q >> lcw;
        node[k] = -1;
        if (q < total && col < un.ncol) {
          const int i = un.col0 + col, iy = div_by(i, inv);
          node[k] = s_node[row] + int64_t(iy) * p.nx + (i - iy * ix);
        }
        old[k] = p.accumulate && node[k] >= 0 ? p.u[node[k]] : 0.0;
      }
#pragma unroll
      for (int k = 0; k < U; ++k) {
        if (node[k] < 0) continue;
        const int q = q0 + k * oz::THREADS, col = c0 + (q & (cw - 1)), row = q >> lcw;
        longlong2 v = make_longlong2(0, 0);
        if (ks == 1) {
          v = sums[col * oz::SUM_PITCH + row];
        } else {
          for (int j = 0; j < ks; ++j) {
            const longlong2 o = *cl.map_shared_rank(sums + col * oz::SUM_PITCH + row, j);
            v.x += o.x;
            v.y += o.y;
          }
        }
        const int er = s_e[row], fc = s_f[col];
        const double y = er == oz::kNonFinite || fc == oz::kNonFinite
                             ? plain_dot(p, p.tiles[p.order[wb.first + row]], un.col0 + col)
                             : oz::sums_to_double(v.x, v.y, er + fc - 62);
        p.u[node[k]] = p.accumulate ? old[k] + y : y;
      }
    }
  }
  if (ks > 1) cl.sync();  // the sums stay until every CTA of the cluster has read them
  oz::release(tmem);
}

constexpr int64_t kMaxWindowBytes = int64_t(1) << 30;  // window digits held at once

}  // namespace

struct OzPlan {
  std::vector<WinBlock> blocks;
  std::vector<Unit> units;
  std::vector<PropRows> rows;
  struct Group { int wb0, nwb, unit0, nunits, ks; };
  std::vector<Group> groups;   // window blocks whose digits are held together
  size_t a_halves = 0, b_halves = 0;
  int ne = 0, nf = 0;
  WinBlock* d_blocks = nullptr;
  Unit* d_units = nullptr;
  PropRows* d_rows = nullptr;
  __half* d_a = nullptr;
  __half* d_b = nullptr;
  int* d_e = nullptr;
  int* d_f = nullptr;
  int* d_err = nullptr;
};

namespace {

// Window blocks, units and groups of a context.
void plan_oz(const lem_ctx* ctx, OzPlan* z) {
  const int nc = int(ctx->classes.size());
  std::vector<int> order(nc);  // classes with many K blocks first: short units fill the tail
  for (int c = 0; c < nc; ++c) order[c] = c;
  auto nkb_of = [&](int c) {
    return (ctx->classes[c].wext[0] * ctx->classes[c].wext[1] + oz::KB - 1) / oz::KB;
  };
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return nkb_of(a) > nkb_of(b); });
  OzPlan::Group g{0, 0, 0, 0, 1};
  int64_t held = 0;
  int ge = 0;
  auto close = [&]() {
    if (g.nwb) z->groups.push_back(g);
    z->a_halves = std::max<size_t>(z->a_halves, size_t(held));
    z->ne = std::max(z->ne, ge);
    g = OzPlan::Group{int(z->blocks.size()), 0, int(z->units.size()), 0, 1};
    held = 0;
    ge = 0;
  };
  for (int c : order) {
    const ClassDesc& cd = ctx->classes[c];
    const int nkb = nkb_of(c), owners = cd.iext[0] * cd.iext[1], ncb = (owners + oz::BN - 1) / oz::BN;
    const int64_t b0 = int64_t(z->b_halves);
    const int f0 = z->nf;
    for (int j = 0; j < ncb; ++j)
      z->rows.push_back(PropRows{c, j * oz::BN, std::min(oz::BN, owners - j * oz::BN),
                                 cd.wext[0] * cd.wext[1], nkb, f0 + j * oz::BN, b0 + int64_t(j) * nkb * oz::B_BLOCK});
    z->b_halves += size_t(ncb) * nkb * oz::B_BLOCK;
    z->nf += ncb * oz::BN;
    const int n0 = ctx->class_offset[c], n1 = ctx->class_offset[c + 1];
    for (int w = n0; w < n1; w += oz::BM) {
      const int64_t halves = int64_t(nkb) * oz::A_BLOCK;
      if (held && (held + halves) * 2 > kMaxWindowBytes) close();
      const int wb = int(z->blocks.size());
      z->blocks.push_back(WinBlock{w, std::min(oz::BM, n1 - w), c, nkb, held, ge, 0});
      held += halves;
      ge += oz::BM;
      g.nwb++;
      for (int j = 0; j < ncb; ++j) {
        z->units.push_back(Unit{wb, j * oz::BN, owners - j * oz::BN, f0 + j * oz::BN, b0 + int64_t(j) * nkb * oz::B_BLOCK});
        g.nunits++;
      }
    }
  }
  close();
}

// CTAs per unit: the split whose estimated time is least, in clk: a K block takes about 1000, a
// unit's set-up and scatter about 8000, a cluster's reduction about 4000 more; `slots` CTAs run
// at once (with clusters, as many as fit beside each other).
int pick_split(const OzPlan::Group& g, const OzPlan* z) {
  double kblocks = 0.0;
  for (int q = 0; q < g.nunits; ++q) kblocks = std::max(kblocks, double(z->blocks[z->units[g.unit0 + q].wb].nkb));
  int best = 1;
  double best_t = 0.0;
  for (int ks : {1, 2, 4, 8}) {
    if (ks > 1 && kblocks / ks < 4) break;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(ks);
    cfg.blockDim = dim3(oz::THREADS);
    cfg.dynamicSmemBytes = oz::SMEM;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = unsigned(ks);
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, oz_step_kernel, &cfg) != cudaSuccess || n < 1) {
      cudaGetLastError();
      if (ks > 1) break;
      n = 152;
    }
    const double waves = std::ceil(double(g.nunits) / n);
    const double t = waves * (kblocks / ks * 1000.0 + 8000.0 + (ks > 1 ? 4000.0 : 0.0));
    if (ks == 1 || t < 0.95 * best_t) {
      best = ks;
      best_t = t;
    }
  }
  return best;
}

}  // namespace

void oz_destroy(lem_ctx* ctx) {
  OzPlan* z = ctx->oz;
  if (!z) return;
  for (void* p : {static_cast<void*>(z->d_blocks), static_cast<void*>(z->d_units), static_cast<void*>(z->d_rows),
                  static_cast<void*>(z->d_a), static_cast<void*>(z->d_b), static_cast<void*>(z->d_e),
                  static_cast<void*>(z->d_f), static_cast<void*>(z->d_err)})
    if (p) cudaFreeAsync(p, ctx->stream);
  delete z;
  ctx->oz = nullptr;
}

// Plan and device memory of the tensor-core FP64 step (at lem_create).
lem_status oz_prepare(lem_ctx* ctx) {
  OzPlan* z = new (std::nothrow) OzPlan();
  if (!z) return fail(LEM_ENOMEM, "host allocation failed");
  ctx->oz = z;
  plan_oz(ctx, z);
  LEM_CUDA_TRY(cudaFuncSetAttribute(oz_step_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, oz::SMEM));
  for (auto& g : z->groups) g.ks = pick_split(g, z);
  auto alloc = [&](auto** p, size_t n) { return dev_alloc(ctx, reinterpret_cast<void**>(p), sizeof(**p) * n); };
  LEM_TRY(alloc(&z->d_blocks, z->blocks.size()));
  LEM_TRY(alloc(&z->d_units, z->units.size()));
  LEM_TRY(alloc(&z->d_rows, z->rows.size()));
  LEM_TRY(alloc(&z->d_b, z->b_halves));
  LEM_TRY(alloc(&z->d_e, size_t(z->ne)));
  LEM_TRY(alloc(&z->d_f, size_t(z->nf)));
  LEM_TRY(alloc(&z->d_err, 1));
  cudaStream_t st = ctx->stream;
  LEM_CUDA_TRY(cudaMemcpyAsync(z->d_blocks, z->blocks.data(), sizeof(WinBlock) * z->blocks.size(),
                               cudaMemcpyHostToDevice, st));
  LEM_CUDA_TRY(cudaMemcpyAsync(z->d_units, z->units.data(), sizeof(Unit) * z->units.size(), cudaMemcpyHostToDevice, st));
  LEM_CUDA_TRY(cudaMemcpyAsync(z->d_rows, z->rows.data(), sizeof(PropRows) * z->rows.size(), cudaMemcpyHostToDevice,
                               st));
  LEM_CUDA_TRY(cudaMemsetAsync(z->d_err, 0, sizeof(int), st));
  return LEM_OK;
}

// Cut the current propagators (after every build, load or adoption, on the context stream).
lem_status oz_pack(lem_ctx* ctx) {
  OzPlan* z = ctx->oz;
  if (!z) return LEM_OK;
  oz_prop_kernel<<<unsigned(z->rows.size() * 8), 256, 0, ctx->stream>>>(ctx->d_P, ctx->n_int, ctx->n_loc, z->d_rows,
                                                                        z->d_f, z->d_b);
  LEM_CUDA_TRY(cudaGetLastError());
  return LEM_OK;
}

lem_status oz_check_error(lem_ctx* ctx) {
  if (!ctx->oz) return LEM_OK;
  int e = 0;
  LEM_CUDA_TRY(cudaMemcpy(&e, ctx->oz->d_err, sizeof(int), cudaMemcpyDeviceToHost));
  if (e == 0) return LEM_OK;
  cudaMemset(ctx->oz->d_err, 0, sizeof(int));
  return fail(LEM_ETIMEOUT, "FP64 tensor-core step gave up waiting on an mbarrier (code " + std::to_string(e) + ")");
}

// One FP64 step; the window digits are allocated at the first.
lem_status step_oz(lem_ctx* ctx, double* d_u) {
  OzPlan* z = ctx->oz;
  cudaStream_t st = ctx->stream;
  if (!z->d_a) {
    LEM_TRY(dev_alloc(ctx, reinterpret_cast<void**>(&z->d_a), sizeof(__half) * z->a_halves));
    // rows past a block's last window are multiplied too (their sums are dropped)
    LEM_CUDA_TRY(cudaMemsetAsync(z->d_a, 0, sizeof(__half) * z->a_halves, st));
  }
  const bool phi = ctx->desc.mode == LEM_MODE_PHI;
  const double* src = d_u;
  if (phi) {
    LEM_CUDA_TRY(launch_residual_fp64(ctx, ctx->d_r, d_u));
    src = ctx->d_r;
  } else {
    // later groups read u^n after earlier ones wrote; so do elements formed in plain FP64
    LEM_CUDA_TRY(cudaMemcpyAsync(ctx->d_r, d_u, sizeof(double) * ctx->npts, cudaMemcpyDeviceToDevice, st));
    src = ctx->d_r;
  }
  cudaEvent_t stop;
  LEM_CUDA_TRY(ctx->timing_begin(&stop));
  for (const OzPlan::Group& g : z->groups) {
    auto cut = g.nwb >= 24 ? oz_windows_kernel<8> : g.nwb >= 12 ? oz_windows_kernel<4> : oz_windows_kernel<2>;
    const int per = g.nwb >= 24 ? 16 : g.nwb >= 12 ? 32 : 64;
    cut<<<unsigned(g.nwb * per), WIN_THREADS, 0, st>>>(src, ctx->d_tiles, ctx->d_class_order, z->d_blocks, g.wb0,
                                                       int(ctx->ny), int(ctx->nx), z->d_e, z->d_a);
    LEM_CUDA_TRY(cudaGetLastError());
    StepParams p{z->d_blocks, z->d_units, ctx->d_tiles, ctx->d_class_order, z->d_a, z->d_b, z->d_e, z->d_f, ctx->d_P,
                 src, d_u, ctx->n_int, ctx->n_loc, ctx->ny, ctx->nx, g.unit0, g.ks, phi ? 1 : 0, z->d_err};
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(unsigned(g.nunits * g.ks));
    cfg.blockDim = dim3(oz::THREADS);
    cfg.dynamicSmemBytes = oz::SMEM;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = unsigned(g.ks);
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    LEM_CUDA_TRY(cudaLaunchKernelEx(&cfg, oz_step_kernel, p));
  }
  ctx->timing_end(stop);
  return LEM_OK;
}

}  // namespace lem
