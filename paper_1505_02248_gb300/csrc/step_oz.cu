// FP64 LEM step on the tensor cores (Sec. 3 steps 1-3, Eq. lem), for contexts whose tiles share
// propagators: exact digit products (oz_core.cuh) in place of FP64 multiply-adds.
//
//   PHI:  r = dt F(u^n); the windows of r, cut into digits (gather and cut in one pass);
//         y = P r|_M for 128 windows x 64 owner rows per CTA; u_D += y.
//   EXP:  the windows of u^n, cut; u_D = P u|_M.
//   Then, in either mode, the owners whose digit sums came out small (settle_cta, oz_small_kernel): a digit
//   sum's error goes with the largest values of the window and of the owner row, so where the values
//   that make up the sum lie far below those, it is formed again as FP64 multiply-adds. Each owner
//   is within 4.1 K 2^-53 sum_k |P_k| |u_k| of its exact sum, as multiply-adds are within K 2^-53 of it; in the
//   mean square the digits are the closer ones (oz::kSmallSum).
//
// GB300's FP64 pipe runs 1.1 TFLOP/s, its FP16 tensor cores 1900. The 1024^2 periodic problem
// (1024 windows of 2304 nodes, 1024 x 2304 propagator) took 4.67 ms a step as one FP64 GEMM, at
// the FP64 pipe's rate, and takes 0.171 ms here (products 110 us, window digits 21, residual 12, small sums
// 20 to 30; the launches chained); a walled 389 x 517 mesh with 16 classes, their GEMMs one
// after another, 29.2 ms a step, and 0.113 ms here. Without the small sums' check it was 0.134 and 0.103 ms.
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
#include <cstdlib>
#include <cstring>
#include <new>
#include <string>
#include <type_traits>
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
  int32_t f0;       // scale exponents of the class's owner rows
  int64_t b0;       // halves into the propagator digits of the class
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

// In place of a scale exponent: a row whose values are all zero (its products are 0).
constexpr int kAllZero = 1 << 21;
// Largest exponent field below which a row is formed in FP64: subnormal values are cut to 0.
constexpr int kTiny = 64;

// A row's scale exponent from the maximum of key_of over its values.
__device__ __forceinline__ int key_of(double v) {  // exponent field, and whether it is not zero
  const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(v));
  return oz::exp_field(b) * 2 + ((b << 1) != 0 ? 1 : 0);
}
__device__ __forceinline__ int exp_of_key(int key) {
  return key == 0 ? kAllZero : key < 2 * kTiny ? oz::kNonFinite : oz::scale_exp(key >> 1);
}

// Magnitudes of eight consecutive values in 8 bits, |x| 2^-e to the nearest 2^-8, from their digits
// (N + kBias). Where a digit sum comes out small, the sum of these times the other operand's tells whether its
// terms are large (a window that changes sign near the owner) or small (a window whose values lie
// orders of magnitude apart).
__device__ __forceinline__ uint2 magnitudes(const unsigned long long (&N)[8]) {
  uint32_t w[2] = {0, 0};
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int n = int(N[u] >> 32) - int(oz::kBias >> 32);  // x 2^-e in units of 2^-23
    w[u / 4] |= min((abs(n) + (1 << 14)) >> 15, 255) << (8 * (u % 4));
  }
  return make_uint2(w[0], w[1]);
}

// Window digits: a CTA cuts R windows of one block (8: one core-matrix row group, so the 16-byte
// stores of 8 lanes fill 128 bytes; fewer where 8 a CTA would leave SMs idle). Its warps find each
// window's largest exponent, then each thread cuts 8 consecutive nodes of one window. Bound by
// the 15 bytes written per node and about 40 integer operations; the two reads of the window come
// from L2. (Eight windows per 256-thread CTA and 64-bit node arithmetic: 43 us for 1024 windows
// of 2304 nodes.)
constexpr int WIN_THREADS = 512;
template <int R>
__global__ void __launch_bounds__(WIN_THREADS) oz_windows_kernel(const double* __restrict__ src,
                                                                 const TileDesc* __restrict__ tiles,
                                                                 const int32_t* __restrict__ order,
                                                                 const WinBlock* __restrict__ blocks, int wb0, int ny,
                                                                 int nx, int* __restrict__ e, __half* __restrict__ out,
                                                                 uint8_t* __restrict__ mag, unsigned* __restrict__ nsmall) {
  constexpr int PER = oz::BM / R;  // CTAs per block
  const WinBlock b = blocks[wb0 + blockIdx.x / PER];
  const int r0 = (blockIdx.x % PER) * R;
  // (chained: the set-up of the multiplying kernel may begin under this one, this one's under the residual)
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (blockIdx.x == 0 && threadIdx.x == 0) *nsmall = 0;
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
      E = max(E, key_of(at(o, a, k - a * wx)));
    }
    for (int q = 16; q > 0; q >>= 1) E = max(E, __shfl_xor_sync(0xffffffffu, E, q));
    if (lane == 0) atomicMax(&ex[r], E);
  }
  __syncthreads();
  const int r = threadIdx.x % R;
  const int sc = exp_of_key(ex[r]);
  if (threadIdx.x < R) e[b.e_off + r0 + r] = sc;
  const int er = sc >= oz::kNonFinite ? 4096 : sc;  // (all zero, or formed in FP64: every digit 0)
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
    *reinterpret_cast<uint2*>(mag + b.a_off / oz::S + size_t(r0 + r) * b.nkb * oz::KB + k8) = magnitudes(N);
  }
}

// Propagator digits, once per build: a CTA cuts 8 owner rows. mid: where the row's largest entries lie.
__global__ void __launch_bounds__(256) oz_prop_kernel(const double* __restrict__ P, int64_t n_int, int64_t n_loc,
                                                      const PropRows* __restrict__ rows, int* __restrict__ f,
                                                      int* __restrict__ mid, uint8_t* __restrict__ mag,
                                                      __half* __restrict__ out) {
  const PropRows p = rows[blockIdx.x / 8];
  const int r0 = (blockIdx.x % 8) * 8;
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  __shared__ int ex[8];
  auto row = [&](int i) { return P + (int64_t(p.cls) * n_int + p.row0 + i) * n_loc; };
  {
    const int fr = p.f_off + r0 + warp, cols = r0 + warp < p.rows ? p.cols : 0;
    const double* P0 = row(r0 + warp);  // (not read past the last row)
    int E = 0;
    for (int k = lane; k < cols; k += 32) E = max(E, key_of(P0[k]));
    for (int o = 16; o > 0; o >>= 1) E = max(E, __shfl_xor_sync(0xffffffffu, E, o));
    int n = 0, at = 0;  // the entries of the largest exponent: their number, the sum of their places
    for (int k = lane; k < cols; k += 32)
      if (key_of(P0[k]) == E) {
        ++n;
        at += k;
      }
    n = __reduce_add_sync(0xffffffffu, n);
    at = __reduce_add_sync(0xffffffffu, at);
    if (lane == 0) {
      f[fr] = ex[warp] = exp_of_key(E);
      mid[fr] = n ? at / n : 0;
    }
  }
  __syncthreads();
  const int r = threadIdx.x % 8;
  const bool live = r0 + r < p.rows;
  const int er = ex[r] >= oz::kNonFinite ? 4096 : ex[r];
  for (int k8 = (threadIdx.x / 8) * 8; k8 < p.nkb * oz::KB; k8 += 256) {
    unsigned long long N[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const double v = live && k8 + u < p.cols ? row(r0 + r)[k8 + u] : 0.0;
      N[u] = oz::biased_digits(static_cast<unsigned long long>(__double_as_longlong(v)), er);
    }
    oz::store_digits(out + p.b_off + size_t(k8 / oz::KB) * oz::B_BLOCK + oz::tile_off(r0 + r, k8 % oz::KB),
                     oz::B_SLICE, N);
    *reinterpret_cast<uint2*>(mag + p.b_off / oz::S + size_t(r0 + r) * p.nkb * oz::KB + k8) = magnitudes(N);
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
  const int* mid;      // where the owner rows' largest entries lie
  const uint8_t* amag; // magnitudes of windows and owner rows
  const uint8_t* bmag;
  const double* P;     // (elements formed in FP64)
  const double* src;
  double* u;
  int64_t n_int, n_loc, ny, nx;
  int unit0, nunits, ks, accumulate;
  int fault;           // test hook (LEM_FAULT=timeout): the first CTA waits for bytes that never come
  int* err;
  unsigned* nsmall;    // elements that oz_small_kernel looks at: their number,
  uint2* small_at;     // window (block * 128 + row) and owner row (its place among the scale exponents; the top
                       // bit: to be formed in any case),
  double* small_old;   // and the owner's value before the step
};

// Per-unit tables of the epilogue.
struct StepTables {
  int2 t0[oz::BM];                    // first owner node of each window
  int e[oz::BM], f[oz::BN];           // scale exponents of the windows, of the owner rows
  int mid[oz::BN];                    // where the owner rows' largest entries lie
  uint32_t in[2], plain[2], zero[2];  // columns (32 a word): owner rows; formed in FP64; all zero
  int ix, wx, wn, oy, ox;             // owners and window nodes per row, window nodes, the owners' place in it
  __device__ void fill(const StepParams& p, const Unit& un, const WinBlock& wb, int t) {
    if (t < 0) return;
    if (t < oz::BM) {
      const TileDesc& d = p.tiles[p.order[wb.first + min(t, wb.count - 1)]];
      t0[t] = make_int2(d.t0[0], d.t0[1]);
      e[t] = t < wb.count ? p.e[wb.e_off + t] : kAllZero;
      if (t == 0) {
        ix = d.iext[1];
        wx = d.wext[1];
        wn = d.wext[0] * wx;
        oy = d.iofs[0];
        ox = d.iofs[1];
      }
    } else if (t < oz::BM + oz::BN) {  // (two whole warps)
      const int c = t - oz::BM, v = p.f[un.f_off + c];
      f[c] = v;
      mid[c] = p.mid[un.f_off + c];
      const uint32_t i = __ballot_sync(0xffffffffu, c < un.ncol);
      const uint32_t q = __ballot_sync(0xffffffffu, v == oz::kNonFinite);
      const uint32_t z = __ballot_sync(0xffffffffu, v == kAllZero);
      if (c % 32 == 0) {
        in[c / 32] = i;
        plain[c / 32] = q;
        zero[c / 32] = z;
      }
    }
  }
};

// Where a unit's outputs go: window by window and owner by owner.
struct StepUnit {
  const StepParams& p;
  const Unit& un;
  const WinBlock& wb;
  const StepTables& t;
  uint32_t inv;          // owners per tile row
  __device__ StepUnit(const StepParams& p_, const Unit& u_, const WinBlock& w_, const StepTables& t_)
      : p(p_), un(u_), wb(w_), t(t_), inv(div_inv(uint32_t(t_.ix))) {}
  __device__ int scale(int row, int col) const { return t.e[row] + t.f[col] - 62; }
  __device__ double value(int, int, double v) const { return v; }
  __device__ int64_t row_at(int row) const {
    return row < wb.count ? int64_t(t.t0[row].x) * p.nx + t.t0[row].y : -1;
  }
  __device__ int64_t col_at(int col) const {
    const int i = un.col0 + col, iy = div_by(i, inv);
    return col < un.ncol ? int64_t(iy) * p.nx + (i - iy * t.ix) : INT64_MIN / 2;
  }
  __device__ double load(int64_t w, int) const { return p.accumulate ? p.u[w] : 0.0; }
  __device__ void store(int64_t w, double y, double old) const { p.u[w] = p.accumulate ? old + y : y; }
  // Of columns 32 h .. 32 h + 31 of a row, those that oz_small_kernel forms in any case: windows or
  // owner rows with infinities, NaN or values too small to cut.
  __device__ uint32_t plain(int row, int h) const {
    return row < wb.count ? (t.e[row] == oz::kNonFinite ? t.in[h] : t.plain[h] & t.in[h]) : 0u;
  }
  // And those that it looks at where their sums are small.
  __device__ uint32_t checked(int row, int h) const {
    return row < wb.count && t.e[row] != kAllZero ? t.in[h] & ~t.zero[h] : 0u;
  }
  // First of the places of this lane's `mine` elements on a list of `count` elements (the whole warp).
  __device__ static uint32_t places(unsigned* count, int mine, int lane) {
    int upto = mine;
#pragma unroll
    for (int o = 1; o < 32; o *= 2) {
      const int v = __shfl_up_sync(0xffffffffu, upto, o);
      if (lane >= o) upto += v;
    }
    unsigned base = 0;
    if (lane == 31 && upto) base = atomicAdd(count, unsigned(upto));
    return __shfl_sync(0xffffffffu, base, 31) + uint32_t(upto - mine);
  }
  __device__ void list(uint32_t place, int row, int col, bool any_case, double old) const {
    p.small_at[place] =
        make_uint2(uint32_t(un.wb) * oz::BM + uint32_t(row), uint32_t(un.f_off + col) | (any_case ? 1u << 31 : 0u));
    if (p.accumulate) p.small_old[place] = old;
  }
};

// The elements that the digits may not give to FP64 accuracy: where the magnitudes of the owner row and of
// the window make sum |P| |u| large, the digit sum stands; 512 nodes around the row's largest entries tell
// as a rule, the others are looked at if they do not (eight lanes per element). Else
// the element is formed as FP64 multiply-adds over the whole row.
// The CTAs of a cluster that shares a unit hold few elements each: they list them in shared memory and look
// at them behind the sums (settle_cta). 256^2, tiles of 16, ten steps 284 us, 327 by oz_small_kernel, whose launch and
// chain of loads take 6 to 9 us a step. CTAs with whole units leave theirs to oz_small_kernel, by a list in
// global memory, of which it takes elements from all over: those of a graded window follow one another
// there, and in their own CTA they would hold up the step (1024^2, four steps 937 us instead of 685; a line of
// 16 384 random values, ten steps, 1156 instead of 345).
// Of the elements of smooth fields 1 to 12 % come here (phi_1 of a residual, mu 50: 39 %), 0 to 0.2 % are
// formed (mu 2, whose rows are narrow: 8 %). Bound by the latency of the loads, or by the FP64 pipe
// where many elements are formed: a step all of whose elements are takes about what it took before it
// used digits (0.9 to 1.1 of it).
constexpr unsigned ALL = 0xffffffffu;
constexpr uint32_t LARGE = 1u << (16 - (38 - oz::kSmallSum));  // 2^-2 in units of 2^-16
// Magnitudes k of the rows at a and b (in 16 bytes): their products, in units of 2^-16.
__device__ __forceinline__ uint32_t magnitude_part(const StepParams& p, uint32_t a, uint32_t b, int k, bool in) {
  if (!in) return 0u;
  const uint4 x = reinterpret_cast<const uint4*>(p.amag)[a + k], y = reinterpret_cast<const uint4*>(p.bmag)[b + k];
  return __dp4a(x.x, y.x, __dp4a(x.y, y.y, __dp4a(x.z, y.z, __dp4a(x.w, y.w, 0u))));
}
__device__ __forceinline__ uint32_t sum_of_eight(uint32_t s) {  // over lanes 8 g .. 8 g + 7
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(ALL, s, o);
  return s;
}
// sum |P| |u| of eight lanes' element, as far as they have to look: nk 16-node parts, the 32 from mid on first.
__device__ __forceinline__ uint32_t magnitude_sum(const StepParams& p, uint32_t a, uint32_t b, int nk, int mid) {
  const int sub = int(threadIdx.x) % 8;
  uint32_t s = 0;
#pragma unroll
  for (int h = 0; h < 4; ++h) s += magnitude_part(p, a, b, mid + sub + 8 * h, mid + sub + 8 * h < nk);
  s = sum_of_eight(s);
  const bool more = s < LARGE && nk > 32;
  if (!__any_sync(ALL, more)) return s;
  uint32_t r = 0;
  if (more) {
#pragma unroll 6
    for (int k = sub; k < nk; k += 8) r += magnitude_part(p, a, b, k, k < mid || k >= mid + 32);
  }
  __syncwarp();
  return s + sum_of_eight(r);
}
__device__ __forceinline__ int middle(int mid, int nk) { return max(min(mid / 16 - 16, nk - 32), 0); }
// The element of an owner row and the window at (oy, ox), wn nodes, wx a row, by LANES lanes of a warp
// (every lane of the warp calls it; wn 0: no element).
template <int LANES>
__device__ __forceinline__ double form(const StepParams& p, const double* row, int oy, int ox, int wx, int wn) {
  const int lane = int(threadIdx.x) % LANES, ny = int(p.ny), nx = int(p.nx);
  const uint32_t inv = div_inv(uint32_t(wx));
  double y = 0.0;
  constexpr int U = 12;  // loads of each operand in flight
  for (int k0 = lane; k0 < wn; k0 += LANES * U) {
    double v[U], w[U];
#pragma unroll
    for (int h = 0; h < U; ++h) {
      const int k = k0 + LANES * h, b = div_by(k, inv);
      int gy = oy + b, gx = ox + (k - b * wx);
      gy = gy < 0 ? gy + ny : (gy >= ny ? gy - ny : gy);
      gx = gx < 0 ? gx + nx : (gx >= nx ? gx - nx : gx);
      v[h] = k < wn ? row[k] : 0.0;
      w[h] = k < wn ? p.src[uint32_t(gy) * uint32_t(nx) + uint32_t(gx)] : 0.0;
    }
#pragma unroll
    for (int h = 0; h < U; ++h) y = fma(v[h], w[h], y);
  }
  __syncwarp();
#pragma unroll
  for (int o = LANES / 2; o > 0; o >>= 1) y += __shfl_xor_sync(ALL, y, o);
  return y;
}
// Calls f with the lanes per element, a constant: eight where `each`, the elements a warp has to form, are more
// than two, so that the sums across lanes (16 clk each of the SM's FP64 pipe, as every FP64 instruction) are
// a small part; a whole warp where they are few and their latency counts. All of a bump's elements, one step:
// 512^2, tiles of 8, 465 -> 332 us (307 with the FP64 GEMM), tiles of 16 1240 -> 827 (846), of 32 2235 -> 2094 (2413).
template <class F>
__device__ __forceinline__ void with_lanes(int each, F f) {
  if (each > 2) f(std::integral_constant<int, 8>());
  else f(std::integral_constant<int, 32>());
}

// A CTA's own list, in shared memory.
struct SmallList {
  double* old;      // the owner's value before the step
  uint16_t* at;     // column * 128 + row; bit 13: to be formed in any case
  uint16_t* todo;   // entries to be formed
  unsigned* count;  // entries; [1]: to be formed
  static constexpr size_t kBytes = 12;  // an entry
  __device__ SmallList(uint8_t* mem, int room, unsigned* n)
      : old(reinterpret_cast<double*>(mem)),
        at(reinterpret_cast<uint16_t*>(old + room)),
        todo(at + room),
        count(n) {}
  __device__ void put(uint32_t place, int row, int col, bool any_case, double before) const {
    old[place] = before;
    at[place] = uint16_t(col * oz::BM + row) | uint16_t(any_case ? 1 << 13 : 0);
  }
};
// Every thread of the CTA calls it, the unit's digit sums written.
__device__ __forceinline__ void settle_cta(const StepUnit& o, const SmallList& l) {
  __syncthreads();
  const int n = int(l.count[0]);
  if (n == 0) return;
  const int warp = int(threadIdx.x) / 32, lane = int(threadIdx.x) % 32, warps = int(blockDim.x) / 32;
  const uint32_t a0 = uint32_t(o.wb.a_off / (16 * oz::S)), b0 = uint32_t(o.wb.b0 / (16 * oz::S));
  for (int i0 = warp * 4; i0 < n; i0 += warps * 4) {
    const int i = i0 + lane / 8, at = i < n ? l.at[i] : 0;
    const int row = at % oz::BM, col = at / oz::BM % oz::BN;
    const bool any_case = at >> 13;
    const int nk = i < n && !any_case ? o.wb.nkb : 0;
    const uint32_t s = magnitude_sum(o.p, a0 + uint32_t(row * o.wb.nkb), b0 + uint32_t(o.un.col0 + col) * uint32_t(o.wb.nkb),
                                     nk, middle(o.t.mid[col], nk));
    if (lane % 8 == 0 && i < n && s < LARGE) l.todo[atomicAdd(l.count + 1, 1u)] = uint16_t(i);
  }
  __syncthreads();
  const int m = int(l.count[1]);
  with_lanes((m + warps - 1) / warps, [&](auto lanes) {
    constexpr int L = decltype(lanes)::value;
    for (int d0 = warp * (32 / L); d0 < m; d0 += warps * (32 / L)) {
      const int d = d0 + lane / L;
      const int i = l.todo[min(d, m - 1)], at = l.at[i], row = at % oz::BM, col = at / oz::BM % oz::BN;
      const double y = form<L>(o.p, o.p.P + (int64_t(o.wb.cls) * o.p.n_int + o.un.col0 + col) * o.p.n_loc,
                               o.t.t0[row].x - o.t.oy, o.t.t0[row].y - o.t.ox, o.t.wx, d < m ? o.t.wn : 0);
      if (d < m && lane % L == 0) o.store(o.row_at(row) + o.col_at(col), y, l.old[i]);
    }
  });
}

constexpr int SMALL_THREADS = 256;
struct Formed {
  int64_t row, to;   // the owner row in P, the owner in the state
  double old;
  int oy, ox, wx, wn;
};
__global__ void __launch_bounds__(SMALL_THREADS, 3) oz_small_kernel(const __grid_constant__ StepParams p) {
  constexpr int WARPS = SMALL_THREADS / 32;
  __shared__ Formed todo[SMALL_THREADS];
  __shared__ int ntodo;
  const int warp = int(threadIdx.x) / 32, lane = int(threadIdx.x) % 32;
  if (threadIdx.x == 0) ntodo = 0;
  __syncthreads();
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int total = int(*p.nsmall), grid = int(gridDim.x);
  for (int64_t first = blockIdx.x; first < total; first += int64_t(SMALL_THREADS) * grid) {
    const int64_t place = first + int64_t(lane * WARPS + warp) * grid;  // (the warps fill evenly)
    const bool valid = place < total;
    const int q = valid ? int(place) : 0;
    // this thread's element
    uint2 at = make_uint2(0, 0);
    int wfirst = 0, i = 0, nk = 0, mid = 0;
    uint32_t oa = 0, ob = 0;  // its magnitudes, in 16 bytes
    bool formed = false;
    if (valid) {
      at = p.small_at[q];
      formed = at.y >> 31;
      at.y &= 0x7fffffffu;
      const WinBlock& wb = p.blocks[at.x / oz::BM];
      wfirst = wb.first;
      i = int(at.y) - wb.f0;
      nk = formed ? 0 : wb.nkb;
      oa = uint32_t(wb.a_off / (16 * oz::S)) + (at.x % oz::BM) * uint32_t(wb.nkb);
      ob = uint32_t(wb.b0 / (16 * oz::S)) + uint32_t(i) * uint32_t(wb.nkb);
      mid = middle(p.mid[at.y], nk);
    }
    // eight lanes per element
    const int g = lane / 8, sub = lane % 8;
    uint32_t sum = 0;
    const unsigned look = __ballot_sync(ALL, nk > 0);
#pragma unroll 1
    for (int e0 = 0; e0 < 32 && look >> e0; e0 += 8) {  // two elements a group
      uint32_t s[2] = {0, 0};
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const int e = e0 + 4 * r + g, m = __shfl_sync(ALL, mid, e) + sub, n = __shfl_sync(ALL, nk, e);
        const uint32_t x = __shfl_sync(ALL, oa, e), y = __shfl_sync(ALL, ob, e);
#pragma unroll
        for (int h = 0; h < 4; ++h) s[r] += magnitude_part(p, x, y, m + 8 * h, m + 8 * h < n);
      }
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        s[r] = sum_of_eight(s[r]);
        s[r] = __shfl_sync(ALL, s[r], (lane % 4) * 8);
        if (lane / 4 == e0 / 4 + r) sum = s[r];
      }
    }
    for (unsigned more = __ballot_sync(ALL, sum < LARGE && nk > 32); more;) {
      int e = -1;  // this group's: the g-th of the next four
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (j == g && more) e = __ffs(int(more)) - 1;
        more &= more - 1;  // (0 stays 0)
      }
      const int l = max(e, 0), m = __shfl_sync(ALL, mid, l), nl = __shfl_sync(ALL, nk, l), n = e < 0 ? 0 : nl;
      const uint32_t x = __shfl_sync(ALL, oa, l), y = __shfl_sync(ALL, ob, l);
      uint32_t s = 0;
#pragma unroll 6
      for (int k = sub; k < n; k += 8) s += magnitude_part(p, x, y, k, k < m || k >= m + 32);
      __syncwarp();
      s = sum_of_eight(s);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int to = __shfl_sync(ALL, e, 8 * j);
        const uint32_t v = __shfl_sync(ALL, s, 8 * j);
        if (lane == to) sum += v;
      }
    }
    if (valid && (formed || sum < LARGE)) {
      const TileDesc& t = p.tiles[p.order[wfirst + int(at.x % oz::BM)]];
      const int iy = i / t.iext[1];
      todo[atomicAdd(&ntodo, 1)] = Formed{(int64_t(t.cls) * p.n_int + i) * p.n_loc,
                                          int64_t(t.t0[0] + iy) * p.nx + t.t0[1] + (i - iy * t.iext[1]),
                                          p.accumulate ? p.small_old[q] : 0.0, t.org[0], t.org[1], t.wext[1],
                                          t.wext[0] * t.wext[1]};
    }
    __syncthreads();
    const int n = ntodo;
    with_lanes((n + WARPS - 1) / WARPS, [&](auto lanes) {
      constexpr int L = decltype(lanes)::value;
      for (int d0 = warp * (32 / L); d0 < n; d0 += WARPS * (32 / L)) {
        const int d = d0 + lane / L;
        const Formed f = todo[min(d, n - 1)];
        const double y = form<L>(p, p.P + f.row, f.oy, f.ox, f.wx, d < n ? f.wn : 0);
        if (d < n && lane % L == 0) p.u[f.to] = p.accumulate ? f.old + y : y;
      }
    });
    __syncthreads();
    if (threadIdx.x == 0) ntodo = 0;
    __syncthreads();
  }
}

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
    return {p.a + wb.a_off, p.b + un.b_off, wb.nkb, p.fault && index(k) == 0};
  }
  __device__ void begin(int k) {
    const Unit& un = p.units[index(k)];
    tab[k & 1].fill(p, un, p.blocks[un.wb], int(threadIdx.x) - 64);
    oz::epi_sync();
  }
  __device__ void finish(int k, int quarter, int half, int lane, double* out, const long long (&hi)[32],
                         const long long (&lo)[32]) {
    const Unit un = p.units[index(k)];
    const WinBlock wb = p.blocks[un.wb];
    const StepUnit o(p, un, wb, tab[k & 1]);
    const int row = 32 * quarter + lane;
    uint32_t small = 0;
#pragma unroll
    for (int j = 0; j < 32; ++j) small |= oz::small_sum(hi[j]) ? 1u << j : 0u;
    const uint32_t plain = o.plain(row, half);
    small = (small & o.checked(row, half)) | plain;
    if (__any_sync(0xffffffffu, small != 0)) {
      uint32_t place = o.places(p.nsmall, __popc(small), lane);
      const int64_t at = o.row_at(row);
#pragma unroll 4
      for (; small; small &= small - 1) {
        const int j = __ffs(int(small)) - 1, col = 32 * half + j;
        o.list(place++, row, col, plain >> j & 1u, o.load(at + o.col_at(col), row));
      }
      __syncwarp();  // (before they are overwritten)
    }
    oz::write_tile(o, quarter, half, lane, out, hi, lo);
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
  __shared__ unsigned s_count[2];
  constexpr size_t SUMS = sizeof(longlong2) * oz::BN * oz::SUM_PITCH;
  static_assert(SUMS % 8 == 0 && SUMS + SmallList::kBytes * oz::BM * oz::BN / 2 <= size_t(oz::STAGES) * oz::STAGE,
                "the list of half the columns fits behind the sums");
  const oz::Shared sh = oz::carve(smem_raw);
  if (threadIdx.x < 2) s_count[threadIdx.x] = 0;
  const int ks = p.ks, rank = int(blockIdx.x) % ks;
  const Unit un = p.units[p.unit0 + int(blockIdx.x) / ks];
  const WinBlock wb = p.blocks[un.wb];
  const uint32_t tmem = oz::setup(sh, &s_abort);
  asm volatile("griddepcontrol.wait;" ::: "memory");  // the window digits are written
  tab.fill(p, un, wb, int(threadIdx.x));
  const int k0 = wb.nkb * rank / ks, k1 = wb.nkb * (rank + 1) / ks;
  SplitWork work{sh, {p.a + wb.a_off + size_t(k0) * oz::A_BLOCK, p.b + un.b_off + size_t(k0) * oz::B_BLOCK, k1 - k0,
                      p.fault && blockIdx.x == 0}};
  oz::run<oz::Fine>(sh, tmem, work, p.err, &s_abort);
  longlong2* sums = reinterpret_cast<longlong2*>(sh.stage);
  cg::cluster_group cl = cg::this_cluster();
  if (k1 == k0)
    for (int q = threadIdx.x; q < oz::BN * oz::SUM_PITCH; q += blockDim.x) sums[q] = make_longlong2(0, 0);
  cl.sync();
  const int lcw = 6 - (31 - __clz(ks)), cw = 1 << lcw, c0 = rank * cw;  // this CTA's columns
  // a CTA that gave up has staged no sums: none of the cluster writes the unit
  bool whole = true;
  for (int j = 0; j < ks; ++j) whole = whole && !*cl.map_shared_rank(const_cast<int*>(&s_abort), j);
  if (whole && c0 < un.ncol) {
    const StepUnit o(p, un, wb, tab);
    const SmallList own(sh.stage + SUMS, oz::BM * oz::BN / 2, s_count);
    constexpr int U = 4;  // elements per thread in flight
    const int total = wb.count * cw, warp0 = int(threadIdx.x) / 32 * 32, lane = int(threadIdx.x) % 32;
    for (int q0 = warp0; q0 < total; q0 += U * oz::THREADS) {  // (whole warps)
      int64_t where[U];
      double old[U];
      bool in[U];
#pragma unroll
      for (int k = 0; k < U; ++k) {
        const int q = q0 + lane + k * oz::THREADS, row = min(q >> lcw, oz::BM - 1);
        const int64_t ra = o.row_at(row), ca = o.col_at(c0 + (q & (cw - 1)));
        in[k] = ra >= 0 && ca >= 0 && q < total;
        where[k] = ra + ca;
        old[k] = in[k] ? o.load(where[k], row) : 0.0;
      }
#pragma unroll
      for (int k = 0; k < U; ++k) {
        const int q = q0 + lane + k * oz::THREADS, col = c0 + (q & (cw - 1)), row = min(q >> lcw, oz::BM - 1);
        longlong2 v = make_longlong2(0, 0);
        if (in[k])
          for (int j = 0; j < ks; ++j) {
            const longlong2 s = *cl.map_shared_rank(sums + col * oz::SUM_PITCH + row, j);
            v.x += s.x;
            v.y += s.y;
          }
        const uint32_t bit = 1u << (col % 32), plain = o.plain(row, col / 32) & bit;
        const bool small = in[k] && (plain || (oz::small_sum(v.x) && (o.checked(row, col / 32) & bit)));
        if (__any_sync(0xffffffffu, small)) {
          const uint32_t place = o.places(own.count, small ? 1 : 0, lane);
          if (small) own.put(place, row, col, plain != 0, old[k]);
        }
        if (in[k]) o.store(where[k], oz::sums_to_double(v.x, v.y, o.scale(row, col)), old[k]);
      }
    }
    settle_cta(o, own);
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
  struct Group {
    int wb0, nwb, unit0, nunits, ks;
    int64_t owners;
  };
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
  int* d_mid = nullptr;
  uint8_t* d_amag = nullptr;
  uint8_t* d_bmag = nullptr;
  unsigned* d_nsmall = nullptr;
  uint2* d_small_at = nullptr;
  double* d_small_old = nullptr;
  int64_t max_owners = 0;      // of a group whose units are not shared
  int fault = 0;
  int64_t bytes = 0;           // device memory of the plan
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
  OzPlan::Group g{0, 0, 0, 0, 1, 0};
  int64_t held = 0;
  int ge = 0;
  auto close = [&]() {
    if (g.nwb) z->groups.push_back(g);
    z->a_halves = std::max<size_t>(z->a_halves, size_t(held));
    z->ne = std::max(z->ne, ge);
    g = OzPlan::Group{int(z->blocks.size()), 0, int(z->units.size()), 0, 1, 0};
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
      z->blocks.push_back(WinBlock{w, std::min(oz::BM, n1 - w), c, nkb, held, ge, f0, b0});
      held += halves;
      g.owners += int64_t(std::min(oz::BM, n1 - w)) * owners;
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
                  static_cast<void*>(z->d_f), static_cast<void*>(z->d_mid), static_cast<void*>(z->d_amag),
                  static_cast<void*>(z->d_bmag), static_cast<void*>(z->d_nsmall),
                  static_cast<void*>(z->d_small_at), static_cast<void*>(z->d_small_old),
                  static_cast<void*>(z->d_err)})
    if (p) cudaFreeAsync(p, ctx->stream);
  ctx->device_bytes -= z->bytes;
  delete z;
  ctx->oz = nullptr;
}

// n elements of the plan's device memory at *p.
template <class T>
static lem_status take(lem_ctx* ctx, T** p, size_t n) {
  const int64_t before = ctx->device_bytes;
  const lem_status s = dev_alloc(ctx, reinterpret_cast<void**>(p), sizeof(T) * n);
  ctx->oz->bytes += ctx->device_bytes - before;
  return s;
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
  for (auto& g : z->groups) {
    g.ks = pick_split(g, z, z->nsm);
    if (g.ks == 1) z->max_owners = std::max(z->max_owners, g.owners);
  }
  LEM_TRY(take(ctx, &z->d_blocks, z->blocks.size()));
  LEM_TRY(take(ctx, &z->d_units, z->units.size()));
  LEM_TRY(take(ctx, &z->d_rows, z->rows.size()));
  LEM_TRY(take(ctx, &z->d_b, z->b_halves));
  LEM_TRY(take(ctx, &z->d_e, size_t(z->ne)));
  LEM_TRY(take(ctx, &z->d_f, size_t(z->nf)));
  LEM_TRY(take(ctx, &z->d_mid, size_t(z->nf)));
  LEM_TRY(take(ctx, &z->d_bmag, z->b_halves / oz::S));
  LEM_TRY(take(ctx, &z->d_nsmall, 1));
  LEM_TRY(take(ctx, &z->d_err, 1));
  const char* fault = std::getenv("LEM_FAULT");
  z->fault = fault && std::strcmp(fault, "timeout") == 0 ? 1 : 0;
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
                                                                        z->d_f, z->d_mid, z->d_bmag, z->d_b);
  LEM_CUDA_TRY(cudaGetLastError());
  return LEM_OK;
}

// (on the context's stream: a plain copy would wait for whatever runs on the legacy stream)
lem_status oz_check_error(lem_ctx* ctx) {
  if (!ctx->oz) return LEM_OK;
  int e = 0;
  LEM_CUDA_TRY(cudaMemcpyAsync(&e, ctx->oz->d_err, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
  LEM_CUDA_TRY(cudaStreamSynchronize(ctx->stream));
  if (e == 0) return LEM_OK;
  cudaMemsetAsync(ctx->oz->d_err, 0, sizeof(int), ctx->stream);
  return fail(LEM_ETIMEOUT, "FP64 tensor-core step gave up waiting on an mbarrier (code " + std::to_string(e) + ")");
}

// Window digits, and room for the list of small sums (at the first step).
static lem_status oz_windows(lem_ctx* ctx) {
  OzPlan* z = ctx->oz;
  if (z->max_owners) LEM_TRY(take(ctx, &z->d_small_at, size_t(z->max_owners)));
  if (z->max_owners && ctx->desc.mode == LEM_MODE_PHI) LEM_TRY(take(ctx, &z->d_small_old, size_t(z->max_owners)));
  LEM_TRY(take(ctx, &z->d_amag, z->a_halves / oz::S));
  LEM_TRY(take(ctx, &z->d_a, z->a_halves));
  // rows past a block's last window are multiplied too (their sums are dropped)
  LEM_CUDA_TRY(cudaMemsetAsync(z->d_a, 0, sizeof(__half) * z->a_halves, ctx->stream));
  return LEM_OK;
}

// One FP64 step. Without room for the window digits the context goes over to the FP64 GEMM, as
// lem_create does without room for those of the propagators.
lem_status step_oz(lem_ctx* ctx, double* d_u) {
  if (!ctx->oz->d_a) {
    const lem_status s = oz_windows(ctx);
    if (s == LEM_ENOMEM) {
      oz_destroy(ctx);
      return step_fp64(ctx, d_u);
    }
    LEM_TRY(s);
  }
  OzPlan* z = ctx->oz;
  cudaStream_t st = ctx->stream;
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
                                    z->d_a, z->d_amag, z->d_nsmall));
    StepParams p{z->d_blocks, z->d_units, ctx->d_tiles, ctx->d_class_order, z->d_a, z->d_b, z->d_e, z->d_f, z->d_mid, z->d_amag, z->d_bmag, ctx->d_P,
                 src, d_u, ctx->n_int, ctx->n_loc, ctx->ny, ctx->nx, g.unit0, g.nunits, g.ks, phi ? 1 : 0, z->fault, z->d_err, z->d_nsmall,
                 z->d_small_at, z->d_small_old};
    if (g.ks == 1) {
      cfg.gridDim = dim3(unsigned(std::min(g.nunits, z->nsm)));
      cfg.blockDim = dim3(oz::THREADS);
      cfg.dynamicSmemBytes = oz::SMEM;
      LEM_CUDA_TRY(cudaLaunchKernelEx(&cfg, oz_step_kernel, p));
    } else {
      cfg = split_config(g.ks, g.nunits, st, at);
      LEM_CUDA_TRY(cudaLaunchKernelEx(&cfg, oz_step_split_kernel, p));
    }
    if (g.ks > 1) continue;
    at[0] = chained();
    cfg.gridDim = dim3(unsigned(3 * z->nsm));
    cfg.blockDim = dim3(SMALL_THREADS);
    cfg.dynamicSmemBytes = 0;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    LEM_CUDA_TRY(cudaLaunchKernelEx(&cfg, oz_small_kernel, p));
  }
  ctx->timing_end(stop);
  return LEM_OK;
}

}  // namespace lem
