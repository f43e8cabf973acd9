// FP64 LEM step on the tensor cores (Sec. 3 steps 1-3, Eq. lem), for contexts whose tiles share
// propagators: exact digit products (oz_core.cuh) in place of FP64 multiply-adds.
//
//   PHI:  r = dt F(u^n); the windows of r, cut into digits (gather and cut in one pass);
//         y = P r|_M for 128 windows x 64 owner rows per CTA; u_D += y.
//   EXP:  the windows of u^n, cut; u_D = P u|_M.
//
// GB300's FP64 pipe runs 1.1 TFLOP/s, its FP16 tensor cores 1900. The 1024^2 periodic problem
// (1024 windows of 2304 nodes, 1024 x 2304 propagator) took 4.67 ms a step as one FP64 GEMM, at
// the FP64 pipe's rate, and takes 0.134 ms here (products 104 us, window digits 20, residual 12, the
// launches chained: 0.141 in a plain sequence); a walled 389 x 517 mesh with 16 classes, their GEMMs one
// after another, 29.2 ms a step, and 0.103 ms here (0.109 unchained).
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
  // (chained: the set-up of the multiplying kernel may begin under this one, this one's under the residual)
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
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

// Owner rows with at most SPARSE nonzero entries (selections, shifts) are formed as FP64
// multiply-adds over those entries, in order: exact where the product with the whole row is,
// whatever the range of the window's values, and cheaper. Their entries are kept with the digits.
constexpr int SPARSE = 8;
constexpr int kSparseRow = 1 << 21;  // in place of the scale exponent

// Propagator digits, once per build: a CTA cuts 8 owner rows.
__global__ void __launch_bounds__(256) oz_prop_kernel(const double* __restrict__ P, int64_t n_int, int64_t n_loc,
                                                      const PropRows* __restrict__ rows, int* __restrict__ f,
                                                      double* __restrict__ sv, int* __restrict__ sk,
                                                      __half* __restrict__ out) {
  const PropRows p = rows[blockIdx.x / 8];
  const int r0 = (blockIdx.x % 8) * 8;
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  __shared__ int ex[8];
  auto row = [&](int i) { return P + (int64_t(p.cls) * n_int + p.row0 + i) * n_loc; };
  {
    int E = 0, cnt = 0;
    const int fr = p.f_off + r0 + warp;
    if (r0 + warp < p.rows)
      for (int k0 = 0; k0 < p.cols; k0 += 32) {
        const int k = k0 + lane;
        const double v = k < p.cols ? row(r0 + warp)[k] : 0.0;
        E = max(E, oz::exp_field(static_cast<unsigned long long>(__double_as_longlong(v))));
        const unsigned nz = __ballot_sync(0xffffffffu, v != 0.0);
        const int at = cnt + __popc(nz & ((1u << lane) - 1u));
        if (v != 0.0 && at < SPARSE) {
          sv[size_t(fr) * SPARSE + at] = v;
          sk[size_t(fr) * SPARSE + at] = k;
        }
        cnt += __popc(nz);
      }
    for (int o = 16; o > 0; o >>= 1) E = max(E, __shfl_xor_sync(0xffffffffu, E, o));
    if (lane < SPARSE && lane >= cnt) sk[size_t(fr) * SPARSE + lane] = -1;
    if (lane == 0) {
      ex[warp] = oz::scale_exp(E);
      f[fr] = ex[warp] != oz::kNonFinite && cnt > 0 && cnt <= SPARSE ? kSparseRow : ex[warp];
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
  const double* sv;    // entries of sparse owner rows
  const int* sk;
  const double* P;     // (rows with infinities or NaN are formed in FP64)
  const double* src;
  double* u;
  int64_t n_int, n_loc, ny, nx;
  int unit0, nunits, ks, accumulate;
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

// The same over the few entries of a sparse owner row.
__device__ __noinline__ double sparse_dot(const StepParams& p, const TileDesc& t, int fr) {
  double s = 0.0;
  for (int q = 0; q < SPARSE; ++q) {
    const int k = p.sk[size_t(fr) * SPARSE + q];
    if (k < 0) break;
    int64_t gy = int64_t(t.org[0]) + k / t.wext[1], gx = int64_t(t.org[1]) + k % t.wext[1];
    gy = gy < 0 ? gy + p.ny : (gy >= p.ny ? gy - p.ny : gy);
    gx = gx < 0 ? gx + p.nx : (gx >= p.nx ? gx - p.nx : gx);
    s = fma(p.sv[size_t(fr) * SPARSE + q], p.src[gy * p.nx + gx], s);
  }
  return s;
}

// Where a unit's outputs go: window by window and owner by owner.
struct StepUnit {
  const StepParams& p;
  Unit un;
  WinBlock wb;
  const int64_t* node0;  // first owner node and scale exponent of each window
  const int* e;
  const int* f;          // scale exponents of the 64 owner rows
  int ix;                // owners per tile row
  uint32_t inv;
  // (rows and columns formed otherwise lie outside for the digit sums: formed() writes them)
  __device__ int scale(int row, int col) const { return e[row] + f[col] - 62; }
  __device__ double value(int, int, double v) const { return v; }
  __device__ int64_t row_at(int row) const { return row < wb.count && e[row] != oz::kNonFinite ? node0[row] : -1; }
  __device__ int64_t off(int col) const {
    const int i = un.col0 + col, iy = div_by(i, inv);
    return int64_t(iy) * p.nx + (i - iy * ix);
  }
  __device__ int64_t col_at(int col) const {
    return col < un.ncol && f[col] != oz::kNonFinite && f[col] != kSparseRow ? off(col) : INT64_MIN / 2;
  }
  // Elements of non-finite windows, non-finite owner rows and sparse owner rows, by this warp:
  // rows r0 .. r0 + nr - 1, columns c0 .. c0 + nc - 1.
  __device__ void formed(int r0, int nr, int c0, int nc, int lane) const {
    bool any = false;
    for (int r = r0 + lane; r < r0 + nr; r += 32) any |= e[r] == oz::kNonFinite;
    for (int c = c0 + lane; c < c0 + nc; c += 32) any |= f[c] == oz::kNonFinite || f[c] == kSparseRow;
    if (!__any_sync(0xffffffffu, any)) return;
    for (int q = lane; q < nr * nc; q += 32) {
      const int row = r0 + q / nc, col = c0 + q % nc;
      if (row >= wb.count || col >= un.ncol) continue;
      const bool plain = e[row] == oz::kNonFinite || f[col] == oz::kNonFinite;
      if (!plain && f[col] != kSparseRow) continue;
      const TileDesc& t = p.tiles[p.order[wb.first + row]];
      const double y = plain ? plain_dot(p, t, un.col0 + col) : sparse_dot(p, t, un.f_off + col);
      const int64_t w = node0[row] + off(col);
      store(w, y, load(w, row));
    }
  }
  __device__ double load(int64_t w, int) const { return p.accumulate ? p.u[w] : 0.0; }
  __device__ void store(int64_t w, double y, double old) const { p.u[w] = p.accumulate ? old + y : y; }
};

// Per-unit tables of the epilogue.
struct StepTables {
  int64_t node0[oz::BM];
  int e[oz::BM], f[oz::BN];
  int ix;
  __device__ void fill(const StepParams& p, const Unit& un, const WinBlock& wb, int t) {
    if (t < oz::BM) {
      const TileDesc& d = p.tiles[p.order[wb.first + min(t, wb.count - 1)]];
      node0[t] = int64_t(d.t0[0]) * p.nx + d.t0[1];
      e[t] = p.e[wb.e_off + t];
      if (t == 0) ix = d.iext[1];
    } else if (t < oz::BM + oz::BN) {
      f[t - oz::BM] = p.f[un.f_off + t - oz::BM];
    }
  }
};

// The units of one CTA, every gridDim.x-th: increments are added to the state (PHI) or the owners
// stored (EXP).
struct StepWork {
  const StepParams& p;
  StepTables* tab;  // [2] by the unit's parity
  __device__ int index(int k) const { return p.unit0 + int(blockIdx.x) + k * int(gridDim.x); }
  __device__ int count() const { return (p.nunits - int(blockIdx.x) + int(gridDim.x) - 1) / int(gridDim.x); }
  __device__ oz::Tile tile(int k) const {
    const Unit& un = p.units[index(k)];
    const WinBlock& wb = p.blocks[un.wb];
    return {p.a + wb.a_off, p.b + un.b_off, wb.nkb};
  }
  __device__ void begin(int k) {
    const Unit& un = p.units[index(k)];
    tab[k & 1].fill(p, un, p.blocks[un.wb], int(threadIdx.x) - 64);
    oz::epi_sync();
  }
  __device__ void finish(int k, int quarter, int half, int lane, double* out, const long long (&hi)[32],
                         const long long (&lo)[32]) {
    const Unit un = p.units[index(k)];
    const StepTables& t = tab[k & 1];
    StepUnit o{p, un, p.blocks[un.wb], t.node0, t.e, t.f, t.ix, div_inv(uint32_t(t.ix))};
    oz::write_tile(o, quarter, half, lane, out, hi, lo);
    o.formed(32 * quarter, 32, 32 * half, 32, lane);
  }
};

__global__ void __launch_bounds__(oz::THREADS, 1) oz_step_kernel(const __grid_constant__ StepParams p) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  __shared__ volatile int s_abort;
  __shared__ StepTables tab[2];
  const oz::Shared sh = oz::carve(smem_raw);
  const uint32_t tmem = oz::setup(sh, &s_abort);
  asm volatile("griddepcontrol.wait;" ::: "memory");  // the window digits are written
  StepWork work{p, tab};
  oz::run<oz::Fine>(sh, tmem, work, p.err, &s_abort);
  oz::release(tmem);
}

// The share of one CTA of a cluster of ks: K blocks [k0, k1) of one unit.
struct SplitWork {
  const oz::Shared& sh;
  oz::Tile t;
  __device__ int count() const { return t.nkb > 0 ? 1 : 0; }
  __device__ oz::Tile tile(int) const { return t; }
  __device__ void begin(int) const {}
  __device__ void finish(int, int quarter, int half, int lane, double*, const long long (&hi)[32],
                         const long long (&lo)[32]) const {
    oz::stage_sums(sh, quarter, half, lane, hi, lo);
  }
};

// One unit per cluster of ks CTAs, its K blocks divided; each CTA then adds the others' sums for
// its share of the columns and writes them.
__global__ void __launch_bounds__(oz::THREADS, 1) oz_step_split_kernel(const __grid_constant__ StepParams p) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  __shared__ volatile int s_abort;
  __shared__ StepTables tab;
  const oz::Shared sh = oz::carve(smem_raw);
  const int ks = p.ks, rank = int(blockIdx.x) % ks;
  const Unit un = p.units[p.unit0 + int(blockIdx.x) / ks];
  const WinBlock wb = p.blocks[un.wb];
  const uint32_t tmem = oz::setup(sh, &s_abort);
  asm volatile("griddepcontrol.wait;" ::: "memory");  // the window digits are written
  tab.fill(p, un, wb, int(threadIdx.x));
  const int k0 = wb.nkb * rank / ks, k1 = wb.nkb * (rank + 1) / ks;
  SplitWork work{sh, {p.a + wb.a_off + size_t(k0) * oz::A_BLOCK, p.b + un.b_off + size_t(k0) * oz::B_BLOCK, k1 - k0}};
  oz::run<oz::Fine>(sh, tmem, work, p.err, &s_abort);
  longlong2* sums = reinterpret_cast<longlong2*>(sh.stage);
  cg::cluster_group cl = cg::this_cluster();
  if (k1 == k0)
    for (int q = threadIdx.x; q < oz::BN * oz::SUM_PITCH; q += blockDim.x) sums[q] = make_longlong2(0, 0);
  cl.sync();
  const int lcw = 6 - (31 - __clz(ks)), cw = 1 << lcw, c0 = rank * cw;  // this CTA's columns
  if (!s_abort && c0 < un.ncol) {
    const StepUnit o{p, un, wb, tab.node0, tab.e, tab.f, tab.ix, div_inv(uint32_t(tab.ix))};
    constexpr int U = 4;  // elements per thread in flight
    const int total = wb.count * cw;
    for (int q0 = threadIdx.x; q0 < total; q0 += U * oz::THREADS) {
      int64_t where[U];
      double old[U];
      bool in[U];
#pragma unroll
      for (int k = 0; k < U; ++k) {
        const int q = q0 + k * oz::THREADS, row = min(q >> lcw, oz::BM - 1);
        const int64_t ra = o.row_at(row), ca = o.col_at(c0 + (q & (cw - 1)));
        in[k] = ra >= 0 && ca >= 0 && q < total;
        where[k] = ra + ca;
        old[k] = in[k] ? o.load(where[k], row) : 0.0;
      }
#pragma unroll
      for (int k = 0; k < U; ++k) {
        if (!in[k]) continue;
        const int q = q0 + k * oz::THREADS, col = c0 + (q & (cw - 1)), row = q >> lcw;
        longlong2 v = make_longlong2(0, 0);
        for (int j = 0; j < ks; ++j) {
          const longlong2 s = *cl.map_shared_rank(sums + col * oz::SUM_PITCH + row, j);
          v.x += s.x;
          v.y += s.y;
        }
        o.store(where[k], oz::sums_to_double(v.x, v.y, o.scale(row, col)), old[k]);
      }
    }
    // (ten warps: 128 / 8 rows for the first eight)
    if (threadIdx.x < 256) o.formed(int(threadIdx.x) / 32 * 16, 16, c0, cw, int(threadIdx.x) % 32);
  }
  cl.sync();  // the sums stay until every CTA of the cluster has read them
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
  int nsm = 152;
  size_t a_halves = 0, b_halves = 0;
  int ne = 0, nf = 0;
  WinBlock* d_blocks = nullptr;
  Unit* d_units = nullptr;
  PropRows* d_rows = nullptr;
  __half* d_a = nullptr;
  __half* d_b = nullptr;
  int* d_e = nullptr;
  int* d_f = nullptr;
  double* d_sv = nullptr;
  int* d_sk = nullptr;
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

// a launch chained to the one ahead of it: the kernel waits for that one itself
cudaLaunchAttribute chained() {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  return at;
}

// at: room for two attributes
cudaLaunchConfig_t split_config(int ks, int units, cudaStream_t st, cudaLaunchAttribute* at) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(unsigned(units * ks));
  cfg.blockDim = dim3(oz::THREADS);
  cfg.dynamicSmemBytes = oz::SMEM;
  cfg.stream = st;
  at->id = cudaLaunchAttributeClusterDimension;
  at->val.clusterDim.x = unsigned(ks);
  at->val.clusterDim.y = at->val.clusterDim.z = 1;
  at[1] = chained();
  cfg.attrs = at;
  cfg.numAttrs = 2;
  return cfg;
}

// CTAs per unit: the split whose estimated time is least, in clk. A K block takes about 1130; a
// unit's share of the scatter that the next unit's MMAs do not cover 3000, set-up and the last
// scatter 12000; with a cluster set-up, reduction and scatter 20000 a wave. As many clusters run
// at once as fit beside each other.
int pick_split(const OzPlan::Group& g, const OzPlan* z, int nsm) {
  double kblocks = 0.0;
  for (int q = 0; q < g.nunits; ++q) kblocks = std::max(kblocks, double(z->blocks[z->units[g.unit0 + q].wb].nkb));
  int best = 1;
  double best_t = std::ceil(double(g.nunits) / nsm) * (kblocks * 1130.0 + 3000.0) + 12000.0;
  for (int ks : {2, 4, 8}) {
    if (kblocks / ks < 4) break;
    cudaLaunchAttribute at[2];
    cudaLaunchConfig_t cfg = split_config(ks, 1, nullptr, at);
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, oz_step_split_kernel, &cfg) != cudaSuccess || n < 1) {
      cudaGetLastError();
      break;
    }
    const double t = std::ceil(double(g.nunits) / n) * (kblocks / ks * 1130.0 + 20000.0);
    if (t < 0.95 * best_t) {
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
                  static_cast<void*>(z->d_f), static_cast<void*>(z->d_sv), static_cast<void*>(z->d_sk),
                  static_cast<void*>(z->d_err)})
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
  LEM_CUDA_TRY(cudaFuncSetAttribute(oz_step_split_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, oz::SMEM));
  if (cudaDeviceGetAttribute(&z->nsm, cudaDevAttrMultiProcessorCount, ctx->device) != cudaSuccess || z->nsm < 1) z->nsm = 152;
  for (auto& g : z->groups) g.ks = pick_split(g, z, z->nsm);
  auto alloc = [&](auto** p, size_t n) { return dev_alloc(ctx, reinterpret_cast<void**>(p), sizeof(**p) * n); };
  LEM_TRY(alloc(&z->d_blocks, z->blocks.size()));
  LEM_TRY(alloc(&z->d_units, z->units.size()));
  LEM_TRY(alloc(&z->d_rows, z->rows.size()));
  LEM_TRY(alloc(&z->d_b, z->b_halves));
  LEM_TRY(alloc(&z->d_e, size_t(z->ne)));
  LEM_TRY(alloc(&z->d_f, size_t(z->nf)));
  LEM_TRY(alloc(&z->d_sv, size_t(z->nf) * SPARSE));
  LEM_TRY(alloc(&z->d_sk, size_t(z->nf) * SPARSE));
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
                                                                        z->d_f, z->d_sv, z->d_sk, z->d_b);
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
    cudaLaunchAttribute at[2] = {chained()};
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(unsigned(g.nwb * per));
    cfg.blockDim = dim3(WIN_THREADS);
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    LEM_CUDA_TRY(cudaLaunchKernelEx(&cfg, cut, src, static_cast<const TileDesc*>(ctx->d_tiles),
                                    static_cast<const int32_t*>(ctx->d_class_order),
                                    static_cast<const WinBlock*>(z->d_blocks), g.wb0, int(ctx->ny), int(ctx->nx), z->d_e,
                                    z->d_a));
    StepParams p{z->d_blocks, z->d_units, ctx->d_tiles, ctx->d_class_order, z->d_a, z->d_b, z->d_e, z->d_f, z->d_sv, z->d_sk, ctx->d_P,
                 src, d_u, ctx->n_int, ctx->n_loc, ctx->ny, ctx->nx, g.unit0, g.nunits, g.ks, phi ? 1 : 0, z->d_err};
    if (g.ks == 1) {
      cfg.gridDim = dim3(unsigned(std::min(g.nunits, z->nsm)));
      cfg.blockDim = dim3(oz::THREADS);
      cfg.dynamicSmemBytes = oz::SMEM;
      LEM_CUDA_TRY(cudaLaunchKernelEx(&cfg, oz_step_kernel, p));
    } else {
      cfg = split_config(g.ks, g.nunits, st, at);
      LEM_CUDA_TRY(cudaLaunchKernelEx(&cfg, oz_step_split_kernel, p));
    }
  }
  ctx->timing_end(stop);
  return LEM_OK;
}

}  // namespace lem
