// FP64 values to and from the digit slices of the tensor-core FP64 products (oz_core.cuh), in
// integer arithmetic only (GB300 runs FP64 at 1/64 of its integer rate). The header compiles
// for the host too, so the arithmetic is checked there bit for bit.
//
// A value |x| < 2^e becomes N = round(x 2^(55 - e)), |N| <= 2^55, and N becomes seven balanced
// base-256 digits, N = sum_s d_s 256^(6 - s), -128 <= d_s <= 127 (d_0 <= 128).
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define LEM_HD __host__ __device__ __forceinline__
#else
#define LEM_HD inline
#endif

namespace lem {
namespace oz {

constexpr int kFracBits = 55;  // N = round(x 2^(55 - e))
// Scale exponent of a row that holds an infinity or a NaN: its products are formed in FP64.
constexpr int kNonFinite = 1 << 20;
// 128 in every digit's place: N + kBias has the digits plus 128, each a plain bit field.
constexpr unsigned long long kBias = 0x0080808080808080ull;

// Biased exponent field of a double's bits (0 for zero and subnormals, which slice to 0).
LEM_HD int exp_field(unsigned long long bits) { return int((bits >> 52) & 0x7FF); }

// Scale exponent from the largest exponent field of a row: every |x| < 2^(E - 1022).
LEM_HD int scale_exp(int E) { return E == 2047 ? kNonFinite : E - 1022; }

// N + kBias for the value with these bits under scale exponent e (not kNonFinite).
LEM_HD unsigned long long biased_digits(unsigned long long bits, int e) {
  const int E = exp_field(bits);
  // x = m 2^(E - 1075) with m in [2^52, 2^53), so N = m 2^(E - 1020 - e), with E - 1022 <= e:
  // a left shift by at most 2, else a rounded right shift (0 beyond the mantissa)
  const int sh = e + 1020 - E;  // right shift, >= -2
  const unsigned long long m = (bits & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull;
  unsigned long long N;
  if (sh <= 0)
    N = m << (sh < -2 ? 2 : -sh);
  else
    N = sh < 54 ? ((m >> (sh - 1)) + 1) >> 1 : 0ull;
  if (E == 0) N = 0;
  if (bits >> 63) N = 0ull - N;
  return N + kBias;
}

// (hi 2^24 + lo) 2^(s) as a double, rounded to nearest even: hi and lo hold the level sums
// sum_{L <= 3} S_L 2^(8 (3 - L)) and sum_{L = 4..6} S_L 2^(8 (6 - L)); |hi| < 2^62, |lo| < 2^62.
LEM_HD double sums_to_double(long long hi, long long lo, int s) {
  long long H = hi + (lo >> 24);
  unsigned int R = (unsigned int)(lo & 0xFFFFFF);  // value = H 2^24 + R
  unsigned long long sign = 0;
  if (H < 0) {  // magnitude
    sign = 1ull << 63;
    H = ~H + (R == 0 ? 1 : 0);
    R = (0x1000000u - R) & 0xFFFFFFu;
  }
  unsigned long long m;  // the magnitude's 64 leading bits
  int ex;                // value = m 2^ex (+ sticky)
  unsigned int sticky = 0;
  if (H == 0) {
    if (R == 0) return 0.0;
#ifdef __CUDA_ARCH__
    const int z = __clz(int(R));
#else
    const int z = __builtin_clz(R);
#endif
    m = (unsigned long long)R << (32 + z);
    ex = -(32 + z);
  } else {
#ifdef __CUDA_ARCH__
    const int z = __clzll(H);
#else
    const int z = __builtin_clzll((unsigned long long)H);
#endif
    m = (unsigned long long)H << z;
    if (z <= 24) {
      m |= R >> (24 - z);
      sticky = R & ((1u << (24 - z)) - 1u);
    } else {
      m |= (unsigned long long)R << (z - 24);
    }
    ex = 24 - z;
  }
  const unsigned int low = (unsigned int)(m & 0x7FF);
  unsigned long long q = m >> 11;  // 53 bits
  const int be = ex + 63 + s + 1023;  // biased exponent of the leading bit
  if (be >= 1) {
    if (low > 0x400u || (low == 0x400u && (sticky != 0 || (q & 1)))) ++q;  // (2^53 carries over)
    unsigned long long b = ((unsigned long long)(unsigned int)(be - 1) << 52) + q;
    if (be >= 2047 || b >= 0x7FF0000000000000ull) b = 0x7FF0000000000000ull;
    b |= sign;
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)b);
#else
    double d;
    __builtin_memcpy(&d, &b, 8);
    return d;
#endif
  }
  // subnormal result: drop 1 - be more bits, rounding once
  const int drop = 12 - be;  // bits of m below the subnormal's unit
  unsigned long long b = 0;
  if (drop <= 64) {
    const unsigned long long top = drop == 64 ? 0ull : m >> drop;
    const unsigned long long half = 1ull << (drop - 1);
    const unsigned long long rest = drop == 64 ? m : m & ((half << 1) - 1);
    b = top;
    if (rest > half || (rest == half && (sticky != 0 || (top & 1)))) ++b;
  }
  b |= sign;
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double d;
  __builtin_memcpy(&d, &b, 8);
  return d;
#endif
}

}  // namespace oz
}  // namespace lem
