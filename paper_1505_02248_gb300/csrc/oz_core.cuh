// FP64 products on the tcgen05 tensor cores: exact sums of FP16 digit products (an Ozaki-type
// splitting), used by the FP64 step (step_oz.cu) and, with coarser digits, by the propagator build
// of the split tiers (builder_tc.cu).
//
// Each row i of A is scaled by 2^-e_i (max |A_i,:| < 2^e_i) and cut into S = 7 balanced digits,
// each column j of B likewise with 2^-f_j. Level L = s + t collects the products of digit s of A
// with digit t of B; levels above 6 are dropped. Every partial sum of a level is an integer of at
// most 24 bits over a bounded stretch of K, which FP32 accumulation holds exactly. After each
// stretch the level sums are drained from TMEM and added up:
//   Fine    base 256 (|d| <= 128, 55 bits and a sign below 2^e_i). Levels 4..6 (at most 7 pairs)
//           over 128 K, levels 0..3 (at most 4) over 256 K; 64-bit integer sums, so
//             C_ij = 2^(e_i + f_j - 62) (hi 2^24 + lo)
//           is exact but for the operands' cut (2^-56 of 2^e_i and of 2^f_j), the dropped levels and the
//           one rounding to FP64. Level 7 is the largest that is dropped, six products of two
//           digits: at most 2^-53.4 of 2^(e_i + f_j) a term, in the mean square 2^-56.3. That is an
//           error by the largest value of a row and of a column, not by the terms of the sum: see
//           kSmallSum for the sums that it does not suit.
//   Coarse  base 128 (49 bits), stretches of 128 K, float-float sums of about 48 bits in the order
//           of the levels: what the FP16 pieces of the split tiers resolve, and cheaper to drain.
// The FP64 pipe (2 multiply-adds per clock and SM) does not take part.
//
// What bounds it: 28 digit products per K. An MMA of N columns takes N / 2 clk but not less than
// its shared-memory operand reads (A 32 clk, B N / 4), 48 clk at N = 64. So one MMA takes digit s
// of A against up to four consecutive digits of B as one operand of 4 x 64 rows: consecutive
// digits of B lie back to back in shared memory, and their products belong to consecutive
// levels, whose accumulators lie back to back in TMEM. Eleven MMAs then do a K step of 16 in 896
// clk (28 of N = 64 take 1344). Measured 1130 clk a K step: shared memory serves 352 clk of A reads,
// 448 of B reads and 336 of the 43 KB that stream in (without the loads 950, without the drains
// 1050, loads alone 720).
#pragma once
#include <cuda_fp16.h>
#include <stdint.h>

#include "oz_convert.h"
#include "tc_ptx.cuh"

namespace lem {
namespace oz {

constexpr int S = 7;      // digits per operand, levels kept
constexpr int BM = 128;   // output rows per CTA (TMEM lanes)
constexpr int BN = 64;    // output columns per CTA
constexpr int KB = 16;    // K elements per block (one MMA K step)
constexpr int A_SLICE = BM * KB;          // halves of one digit's tile
constexpr int B_SLICE = BN * KB;
constexpr int A_BLOCK = S * A_SLICE;      // halves of one K block, all digits
constexpr int B_BLOCK = S * B_SLICE;
constexpr int A_BYTES = A_BLOCK * 2;      // 28 KB
constexpr int B_BYTES = B_BLOCK * 2;      // 14 KB
constexpr int STAGE = A_BYTES + B_BYTES;
constexpr int STAGES = 5;                 // 215 KB of the SM's 227
constexpr int STRETCH_LO = 8;             // K blocks per exact stretch of levels 4..6 (128 K)
constexpr int GROUP = 4;                  // K blocks whose levels 0..3 go before their levels 4..6
constexpr int EPI_WARPS = 8;              // two per TMEM lane quarter, 32 columns each
constexpr int THREADS = 64 + 32 * EPI_WARPS;
constexpr int OUT_PITCH = 5;               // doubles per row of a warp's output chunk (4 columns)
constexpr int OUT_BYTES = EPI_WARPS * 32 * OUT_PITCH * 8;
constexpr int SMEM = STAGES * STAGE + OUT_BYTES + 1024 + 256;
constexpr uint64_t WAIT_NS = 2000000000ull;
constexpr int SUM_PITCH = BM + 1;         // staged sums: column pitch in 16-byte (hi, lo) pairs
// Fine sums |C_ij| below 2^-2 of 2^(e_i + f_j), |hi| below 2^36, are small: unless their terms are known
// to be large (sum_k |A_ik| |B_kj| at least that), FP64 multiply-adds are closer to the true sum, and
// the caller forms them so. The line is where the two errors cross. Root mean squares of digits
// over multiply-adds on windows of the phi_1 and exponential propagators (K 96 .. 2304), by that sum
// of magnitudes over 2^(e_i + f_j): in [1/16, 1/8) 3.2, [1/8, 1/4) 1.1 .. 1.5, [1/4, 1/2) 0.75 .. 1.3,
// [1/2, 1) 0.36 .. 0.84, above 1 0.56 .. 0.03.
constexpr int kSmallSum = 36;

static_assert(STRETCH_LO % GROUP == 0 && GROUP < STAGES, "groups end stretches");
static_assert(BN * SUM_PITCH * 16 <= STAGES * STAGE, "staged sums reuse the operand stages");

// Operand tiles: for each block of 128 (A) or 64 (B) rows and each K block of 16, the seven
// digits' tiles back to back. A tile is in the tcgen05 K-major layout without swizzle: 8-row x
// 8-element core matrices of 128 contiguous bytes, two along K (128 B apart), 8-row groups 256 B
// apart. So element (r, k) of a tile sits at half offset (r / 8) 128 + (k / 8) 64 + (r % 8) 8 + k % 8.
__device__ __forceinline__ int tile_off(int r, int k8) {  // k8: first of 8 consecutive K elements
  return (r / 8) * 128 + (k8 / 8) * 64 + (r % 8) * 8;
}

// The seven digits of 8 consecutive K elements (as N + kBias) into their tiles: `dst` is the
// element's place in digit 0's tile, tiles lie `slice` halves apart.
__device__ __forceinline__ void store_digits(__half* dst, int slice, const unsigned long long (&N)[8]) {
  uint32_t lo[8], hi[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    lo[u] = uint32_t(N[u]);
    hi[u] = uint32_t(N[u] >> 32);
  }
  const __half2 bias = __half2half2(__ushort_as_half(0x6480));  // 1024 + 128
#pragma unroll
  for (int s = 0; s < S; ++s) {
    uint32_t w[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      uint32_t t;
      if (s == 0) {  // the top field has nine bits (0 .. 256)
        t = ((hi[2 * q] >> 16) & 0x1FFu) + ((hi[2 * q + 1] & 0x1FF0000u)) + 0x64006400u;
      } else {
        const int byte = 6 - s;  // place of digit s in N
        const uint32_t a = byte >= 4 ? hi[2 * q] : lo[2 * q], b = byte >= 4 ? hi[2 * q + 1] : lo[2 * q + 1];
        const uint32_t sel = uint32_t(byte & 3) | (uint32_t(4 + (byte & 3)) << 8);
        t = __byte_perm(a, b, (sel & 0xF) | ((sel >> 8) << 8));
        t = (t & 0x00FF00FFu) | 0x64006400u;
      }
      // 1024 + (digit + 128) as a half, minus 1152: the digit, exactly
      const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&t), bias);
      w[q] = *reinterpret_cast<const uint32_t*>(&h);
    }
    *reinterpret_cast<uint4*>(dst + s * slice) = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

// The same for coarse digits, given as integers.
__device__ __forceinline__ void store_coarse_digits(__half* dst, int slice, const int (&d)[8][S]) {
  const __half2 bias = __half2half2(__ushort_as_half(0x6480));  // 1024 + 128
#pragma unroll
  for (int s = 0; s < S; ++s) {
    uint32_t w[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const uint32_t t = uint32_t(d[2 * q][s] + 128) + (uint32_t(d[2 * q + 1][s] + 128) << 16) + 0x64006400u;
      const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&t), bias);
      w[q] = *reinterpret_cast<const uint32_t*>(&h);
    }
    *reinterpret_cast<uint4*>(dst + s * slice) = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

// Shared-memory layout of a CTA, and its barriers.
struct Shared {
  uint8_t* stage;   // STAGES x STAGE bytes
  double* out;      // [EPI_WARPS][32][OUT_PITCH] output chunks
  uint64_t* full;   // [STAGES] stage loaded
  uint64_t* empty;  // [STAGES] stage consumed by the MMAs
  uint64_t* accf;   // [2] levels 0..3 / 4..6 complete for a stretch
  uint64_t* acce;   // [2] drained
  uint32_t* tslot;
};

__device__ __forceinline__ Shared carve(uint8_t* raw) {
  Shared sh;
  // (offset arithmetic on the shared array keeps the pointers in the shared address space)
  sh.stage = raw + ((1024u - (ptx::smem_u32(raw) & 1023u)) & 1023u);
  sh.out = reinterpret_cast<double*>(sh.stage + STAGES * STAGE);
  uint64_t* bars = reinterpret_cast<uint64_t*>(sh.stage + STAGES * STAGE + OUT_BYTES);
  sh.full = bars;
  sh.empty = bars + STAGES;
  sh.accf = bars + 2 * STAGES;
  sh.acce = sh.accf + 2;
  sh.tslot = reinterpret_cast<uint32_t*>(sh.acce + 2);
  return sh;
}

// Barriers and TMEM (all 512 columns: 448 hold the levels); every thread of the CTA calls it.
__device__ __forceinline__ uint32_t setup(const Shared& sh, volatile int* s_abort) {
  if (threadIdx.x == 0) {
    *s_abort = 0;
    for (int q = 0; q < STAGES; ++q) {
      ptx::mbar_init(&sh.full[q], 1);
      ptx::mbar_init(&sh.empty[q], 1);
    }
    for (int h = 0; h < 2; ++h) {
      ptx::mbar_init(&sh.accf[h], 1);
      ptx::mbar_init(&sh.acce[h], EPI_WARPS);
    }
    ptx::fence_barrier_init();
  }
  if (threadIdx.x / 32 == 1) {
    ptx::tmem_alloc(sh.tslot, 512);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  return *sh.tslot;
}

__device__ __forceinline__ void release(uint32_t tmem) {
  ptx::tc_fence_before();
  __syncthreads();
  if (threadIdx.x / 32 == 1) {
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem, 512);
  }
}

// Levels [L0, L0 + n) of 32 columns of this thread's row, in order, to add(L, column, sum); the next
// 16 columns load while these are added.
template <int L0, int n, class Add>
__device__ __forceinline__ void drain(uint32_t base, Add add) {
  uint32_t r[2][16];
  ptx::tmem_issue_x16(base + L0 * BN, r[0]);
#pragma unroll
  for (int q = 0; q < 2 * n; ++q) {
    ptx::tmem_wait_x16(r[q & 1]);
    if (q + 1 < 2 * n)
      ptx::tmem_issue_x16(base + uint32_t((L0 + (q + 1) / 2) * BN + 16 * ((q + 1) & 1)), r[(q + 1) & 1]);
#pragma unroll
    for (int j = 0; j < 16; ++j) add(L0 + q / 2, 16 * (q & 1) + j, __uint_as_float(r[q & 1][j]));
  }
}

struct Fine {
  using Acc = long long;
  static constexpr int STRETCH_HI = 16;  // K blocks per exact stretch of levels 0..3 (256 K)
  static __device__ __forceinline__ void drain_hi(uint32_t base, Acc (&hi)[32], Acc (&)[32]) {
    drain<0, 4>(base, [&](int L, int j, float x) { hi[j] += (long long)(__float2int_rn(x)) * (1 << (8 * (3 - L))); });
  }
  static __device__ __forceinline__ void drain_lo(uint32_t base, Acc (&)[32], Acc (&lo)[32]) {
    drain<4, 3>(base, [&](int L, int j, float x) { lo[j] += (long long)(__float2int_rn(x)) * (1 << (8 * (6 - L))); });
  }
};

struct Coarse {
  using Acc = float;
  static constexpr int STRETCH_HI = STRETCH_LO;
  static __device__ __forceinline__ void ff_add(float& hi, float& lo, float x) {
    const float s = __fadd_rn(hi, x);
    const float bb = __fsub_rn(s, hi);
    const float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(x, bb));
    hi = s;
    lo = __fadd_rn(lo, e);
  }
  // sum_L S_L 2^-7L in float-float
  template <int L0, int n>
  static __device__ __forceinline__ void drain_any(uint32_t base, Acc (&hi)[32], Acc (&lo)[32]) {
    drain<L0, n>(base, [&](int L, int j, float x) {
      ff_add(hi[j], lo[j], __fmul_rn(x, __int_as_float((127 - 7 * L) << 23)));
    });
  }
  static __device__ __forceinline__ void drain_hi(uint32_t base, Acc (&hi)[32], Acc (&lo)[32]) {
    drain_any<0, 4>(base, hi, lo);
  }
  static __device__ __forceinline__ void drain_lo(uint32_t base, Acc (&hi)[32], Acc (&lo)[32]) {
    drain_any<4, 3>(base, hi, lo);
  }
  // (hi + lo) 2^E: the scaled doubles come from the float bits, leaving one FP64 addition
  static __device__ __forceinline__ double f32_scaled(float x, int E) {
    const uint32_t b = __float_as_uint(x);
    const int e8 = static_cast<int>((b >> 23) & 0xFF);
    const int ed = e8 - 127 + E + 1023;
    unsigned long long v = (static_cast<unsigned long long>(ed) << 52) | (static_cast<unsigned long long>(b & 0x7FFFFF) << 29);
    v = ed >= 2047 ? 0x7FF0000000000000ull : v;
    v |= static_cast<unsigned long long>(b >> 31) << 63;
    return __longlong_as_double(static_cast<long long>(e8 == 0 || ed <= 0 ? 0ull : v));
  }
  static __device__ __forceinline__ double value(float hi, float lo, int E) { return f32_scaled(hi, E) + f32_scaled(lo, E); }
};

// One unit of work: the digit products of nkb K blocks (nkb >= 1) of one 128 x 64 output tile.
struct Tile {
  const __half* a;  // the tile's first K block
  const __half* b;
  int nkb;
  bool stall = false;  // test hook: its first stage is armed, but not all of its bytes are loaded
};

// Barrier among the epilogue warps.
__device__ __forceinline__ void epi_sync() { asm volatile("bar.sync 1, %0;" ::"n"(32 * EPI_WARPS) : "memory"); }

// The CTA's units, one after another: warp 0 loads, warp 1 issues the MMAs, warps 2..9 drain and
// write: thread = output row (TMEM lane), 32 of its 64 columns. While the epilogue warps write a
// tile, the MMAs of the next one already run, up to the end of its first stretches. Work:
//   int count()                     units of this CTA
//   Tile tile(int k)                unit k (every role asks for it)
//   void begin(int k)               epilogue threads, before unit k's sums are drained (may hold an
//                                   epi_sync: each of them calls it for every unit)
//   void finish(int k, quarter, half, lane, out, hi, lo)   its sums: hi, lo of the thread's columns
// Mode: Fine or Coarse sums.
// Every thread of the CTA calls it; a barrier ends it. A wait that runs out records `err`, sets
// s_abort and lets the CTA finish without writing.
template <class Mode, class Work>
__device__ __forceinline__ void run(const Shared& sh, uint32_t tmem, Work& work, int* err, volatile int* s_abort) {
  constexpr int STRETCH_HI = Mode::STRETCH_HI;
  static_assert(STRETCH_HI == STRETCH_LO || STRETCH_HI == 2 * STRETCH_LO, "drained with every or every second low stretch");
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int count = work.count();
  if (warp == 0) {
    if (lane == 0) {
      int issued = 0, q = 0;
      uint32_t par = 0;
      for (int k = 0; k < count && !*s_abort; ++k) {
        const Tile t = work.tile(k);
        for (int kb = 0; kb < t.nkb && !*s_abort; ++kb) {
          if (issued >= STAGES && !ptx::mbar_wait(&sh.empty[q], par ^ 1u, WAIT_NS)) {
            atomicExch(err, 1);
            *s_abort = 1;
            break;
          }
          uint8_t* st = sh.stage + q * STAGE;
          ptx::mbar_arrive_expect_tx(&sh.full[q], STAGE);
          ptx::bulk_load(st, t.a + size_t(kb) * A_BLOCK, A_BYTES, &sh.full[q]);
          if (!t.stall || kb) ptx::bulk_load(st + A_BYTES, t.b + size_t(kb) * B_BLOCK, B_BYTES, &sh.full[q]);
          ++issued;
          if (++q == STAGES) {
            q = 0;
            par ^= 1u;
          }
        }
      }
      // every copy issued has landed before the CTA reuses the stages or exits
      for (int kb = issued > STAGES ? issued - STAGES : 0; kb < issued; ++kb)
        ptx::mbar_wait(&sh.full[kb % STAGES], (kb / STAGES) & 1, WAIT_NS);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      // K blocks are taken four at a time, first their products of levels 0..3, then those of
      // levels 4..6: while one group of levels is drained the MMAs of the other group run (one K
      // block at a time, the drains held the MMAs up: 1360 clk a K block).
      constexpr uint64_t SA = A_SLICE * 2 / 16, SB = B_SLICE * 2 / 16;  // descriptor steps per digit
      const uint32_t s0 = ptx::smem_u32(sh.stage);
      const uint64_t dA0 = ptx::plain_kmajor_desc(s0, 128, 256), dB0 = ptx::plain_kmajor_desc(s0 + A_BYTES, 128, 256);
      bool ok = true;
      int qa = 0, qb = 0, nhi = 0, nlo = 0;  // stretches begun
      uint32_t par = 0;
      for (int k = 0; k < count && ok; ++k) {
        const int nkb = work.tile(k).nkb;
        for (int k0 = 0; k0 < nkb && ok; k0 += GROUP) {
          const int k1 = k0 + GROUP < nkb ? k0 + GROUP : nkb;
          if (k0 % STRETCH_HI == 0 && nhi++ > 0) {  // (drained up to the stretch before)
            if (!ptx::mbar_wait(&sh.acce[0], (nhi - 2) & 1, WAIT_NS)) { ok = false; break; }
          }
          for (int kb = k0; kb < k1; ++kb) {
            if (!ptx::mbar_wait(&sh.full[qa], par, WAIT_NS)) { ok = false; break; }
            ptx::tc_fence_after();
            const uint64_t dA = dA0 + uint64_t(qa * (STAGE >> 4)), dB = dB0 + uint64_t(qa * (STAGE >> 4));
            // digit s of A against digits 0 .. 3 - s of B
            ptx::mma_f16(tmem, dA, dB, ptx::idesc_f16_f32(BM, 4 * BN), kb % STRETCH_HI == 0 ? 0u : 1u);
            ptx::mma_f16(tmem + BN, dA + SA, dB, ptx::idesc_f16_f32(BM, 3 * BN), 1u);
            ptx::mma_f16(tmem + 2 * BN, dA + 2 * SA, dB, ptx::idesc_f16_f32(BM, 2 * BN), 1u);
            ptx::mma_f16(tmem + 3 * BN, dA + 3 * SA, dB, ptx::idesc_f16_f32(BM, BN), 1u);
            if (++qa == STAGES) {
              qa = 0;
              par ^= 1u;
            }
          }
          if (!ok) break;
          if (k1 % STRETCH_HI == 0 || k1 == nkb) ptx::mma_commit(&sh.accf[0]);
          if (k0 % STRETCH_LO == 0 && nlo++ > 0) {
            if (!ptx::mbar_wait(&sh.acce[1], (nlo - 2) & 1, WAIT_NS)) { ok = false; break; }
            ptx::tc_fence_after();
          }
          for (int kb = k0; kb < k1; ++kb) {
            const uint64_t dA = dA0 + uint64_t(qb * (STAGE >> 4)), dB = dB0 + uint64_t(qb * (STAGE >> 4));
            // digit s of A against digits max(4 - s, 0) .. 6 - s of B
            ptx::mma_f16(tmem + 4 * BN, dA, dB + 4 * SB, ptx::idesc_f16_f32(BM, 3 * BN),
                         kb % STRETCH_LO == 0 ? 0u : 1u);
#pragma unroll
            for (int s = 1; s < 5; ++s)
              ptx::mma_f16(tmem + 4 * BN, dA + s * SA, dB + (4 - s) * SB, ptx::idesc_f16_f32(BM, 3 * BN), 1u);
            ptx::mma_f16(tmem + 5 * BN, dA + 5 * SA, dB, ptx::idesc_f16_f32(BM, 2 * BN), 1u);
            ptx::mma_f16(tmem + 6 * BN, dA + 6 * SA, dB, ptx::idesc_f16_f32(BM, BN), 1u);
            ptx::mma_commit(&sh.empty[qb]);
            if (++qb == STAGES) qb = 0;
          }
          if (k1 % STRETCH_LO == 0 || k1 == nkb) ptx::mma_commit(&sh.accf[1]);
        }
      }
      if (!ok) {
        atomicExch(err, 2);
        *s_abort = 1;
      }
    }
  } else {
    const int e = warp - 2, quarter = warp & 3, half = e >> 2;
    const uint32_t base = tmem + (uint32_t(32 * quarter) << 16) + uint32_t(32 * half);
    bool ok = true;
    uint32_t phi = 0, plo = 0;  // phases of accf
    for (int k = 0; k < count; ++k) {  // (to the end also after a failed wait: begin() has a barrier)
      typename Mode::Acc hi[32], lo[32];
#pragma unroll
      for (int j = 0; j < 32; ++j) hi[j] = lo[j] = 0;
      work.begin(k);
      const int nlo = (work.tile(k).nkb + STRETCH_LO - 1) / STRETCH_LO;
      for (int c = 0; c < nlo && ok; ++c) {
        if (STRETCH_HI == STRETCH_LO || (c & 1) || c == nlo - 1) {  // levels 0..3 end a stretch of theirs
          if (*s_abort || !ptx::mbar_wait(&sh.accf[0], phi, WAIT_NS)) { ok = false; break; }
          phi ^= 1u;
          ptx::tc_fence_after();
          Mode::drain_hi(base, hi, lo);
          ptx::tc_fence_before();
          __syncwarp();
          if (lane == 0) ptx::mbar_arrive(&sh.acce[0]);
        }
        if (*s_abort || !ptx::mbar_wait(&sh.accf[1], plo, WAIT_NS)) { ok = false; break; }
        plo ^= 1u;
        ptx::tc_fence_after();
        Mode::drain_lo(base, hi, lo);
        ptx::tc_fence_before();
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(&sh.acce[1]);
      }
      if (ok) work.finish(k, quarter, half, lane, sh.out + e * 32 * OUT_PITCH, hi, lo);
    }
    if (!ok && lane == 0) {
      atomicExch(err, 3);
      *s_abort = 1;
    }
  }
  __syncthreads();
}

// Whether a fine sum is small (kSmallSum); levels 4..6 are below 2^22.
__device__ __forceinline__ bool small_sum(long long hi) {
  return unsigned(int(hi >> 32) + (1 << (kSmallSum - 32))) < (2u << (kSmallSum - 32));
}
// The usual finish: each thread's sums as doubles, passed through the warp's output chunk four
// columns at a time, so that 4 lanes write 32 consecutive bytes of a row. Out:
//   int scale(row, col)                  the element is its sums times 2^scale
//   double value(row, col, v)            what is passed on of the scaled sum v
//   int64_t row_at(row), col_at(col)     an element's place is their sum; negative: outside
//   double load(row_at + col_at, row)    the old value (loaded a chunk ahead)
//   void store(place, value, old)
template <class Out, class Acc>
__device__ __forceinline__ void write_tile(const Out& o, int quarter, int half, int lane, double* out,
                                           const Acc (&hi)[32], const Acc (&lo)[32]) {
  const int row = 32 * quarter + lane;
  const int r8 = lane / 4, c4 = lane % 4;
  int64_t ra[4];
  bool rin[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    ra[r] = o.row_at(32 * quarter + 8 * r + r8);
    rin[r] = ra[r] >= 0;
  }
  double old[2][4];
  int64_t ca[2];
  bool cin[2];
  auto fetch = [&](int t) {
    ca[t & 1] = o.col_at(32 * half + 4 * t + c4);
    cin[t & 1] = ca[t & 1] >= 0;
#pragma unroll
    for (int r = 0; r < 4; ++r)
      old[t & 1][r] = rin[r] && cin[t & 1] ? o.load(ra[r] + ca[t & 1], 32 * quarter + 8 * r + r8) : 0.0;
  };
  fetch(0);
#pragma unroll
  for (int t = 0; t < 8; ++t) {
    if (t < 7) fetch(t + 1);
    double y[4];
    if constexpr (sizeof(Acc) == 4) {
#pragma unroll
      for (int q = 0; q < 4; ++q)
        y[q] = Coarse::value(hi[4 * t + q], lo[4 * t + q], o.scale(row, 32 * half + 4 * t + q));
    } else {
      double v[4];
      bool far = false;
#pragma unroll
      for (int q = 0; q < 4; ++q) v[q] = sums_unscaled(hi[4 * t + q], lo[4 * t + q]);
#pragma unroll
      for (int q = 0; q < 4; ++q) y[q] = scale_near(v[q], o.scale(row, 32 * half + 4 * t + q) + 24, &far);
      if (__any_sync(0xffffffffu, far)) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          bool f = false;
          const int s = o.scale(row, 32 * half + 4 * t + q) + 24;
          scale_near(v[q], s, &f);
          if (f) y[q] = scale_far(v[q], s);
        }
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) out[lane * OUT_PITCH + q] = o.value(row, 32 * half + 4 * t + q, y[q]);
    __syncwarp();
#pragma unroll
    for (int r = 0; r < 4; ++r)
      if (rin[r] && cin[t & 1]) o.store(ra[r] + ca[t & 1], out[(8 * r + r8) * OUT_PITCH + c4], old[t & 1][r]);
    __syncwarp();
  }
}

// The sums in shared memory, over the operand stages (the last unit only: every load has then
// been consumed): pair (hi, lo) of element (row, col) at [col * SUM_PITCH + row].
__device__ __forceinline__ void stage_sums(const Shared& sh, int quarter, int half, int lane,
                                           const long long (&hi)[32], const long long (&lo)[32]) {
  longlong2* sums = reinterpret_cast<longlong2*>(sh.stage);
#pragma unroll
  for (int j = 0; j < 32; ++j)
    sums[(32 * half + j) * SUM_PITCH + 32 * quarter + lane] = make_longlong2(hi[j], lo[j]);
}

}  // namespace oz
}  // namespace lem
