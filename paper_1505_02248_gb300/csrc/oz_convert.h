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

// Coarse digits: N = round(x 2^(49 - e)), |N| <= 2^49, as seven balanced base-128 digits, each
// rounded to nearest from the top (|d_0| <= 128, the others at most 64 in magnitude).
LEM_HD void coarse_digits(unsigned long long bits, int e, int (&d)[7]) {
  const int E = exp_field(bits);
  const int sh = 1026 + e - E;  // >= 4
  long long N = 0;
  if (E != 0 && sh < 54) {
    const long long m = (long long)((bits & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull);
    N = (m + (1ll << (sh - 1))) >> sh;
    if (bits >> 63) N = -N;
  }
  for (int s = 0; s < 6; ++s) {
    const int p = 7 * (6 - s);
    const long long q = (N + (1ll << (p - 1))) >> p;  // arithmetic shift: floor
    N -= q << p;
    d[s] = (int)q;
  }
  d[6] = (int)N;
}

LEM_HD double bits_double(unsigned long long b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double d;
  __builtin_memcpy(&d, &b, 8);
  return d;
#endif
}
LEM_HD unsigned long long double_bits(double d) {
#ifdef __CUDA_ARCH__
  return (unsigned long long)__double_as_longlong(d);
#else
  unsigned long long b;
  __builtin_memcpy(&b, &d, 8);
  return b;
#endif
}

// Largest K of a product: the level sums stay below 2^51 2^24.
constexpr int kMaxK = 8000;

// (hi 2^24 + lo) 2^s as a double, rounded to nearest even (twice if it is subnormal): hi and lo
// hold the level sums sum_{L <= 3} S_L 2^(8 (3 - L)) and sum_{L = 4..6} S_L 2^(8 (6 - L));
// |hi + (lo >> 24)| < 2^51. Two FP64 additions, the first exact: H = hi + (lo >> 24) enters as
// the low mantissa bits of 1.5 2^52, the 24 bits below it as 1 + R 2^-24, and the integers need no
// conversion instructions. (All in integers it took about 80 instructions an element, and the
// epilogue of a tile 22 us.)
LEM_HD double sums_unscaled(long long hi, long long lo) {  // (hi 2^24 + lo) 2^-24
  const long long H = hi + (lo >> 24);
  const unsigned long long R = (unsigned long long)lo & 0xFFFFFFull;
  const double h = bits_double((unsigned long long)H + 0x4338000000000000ull) - 6755399441055745.0;  // H - 1
  return h + bits_double(0x3FF0000000000000ull | (R << 28));
}
// v 2^t where v and the result are normal numbers or v is zero; *far is set where they are not.
// No branches, so that several elements' instructions interleave.
LEM_HD double scale_near(double v, int t, bool* far) {
  const unsigned long long b = double_bits(v);
  const unsigned int e = (unsigned int)((b >> 52) & 0x7FF);
  const bool zero = e == 0;  // (an FP64 comparison would cost as much as an addition)
  *far = *far || (!zero && (unsigned int)((int)e + t - 1) >= 2046u);
  return bits_double(zero ? b : b + ((unsigned long long)(unsigned int)t << 52));
}
LEM_HD double scale_far(double v, int t) {  // in three steps, of which the last one rounds
  const int q = t / 3;
  const double f = bits_double((unsigned long long)(1023 + q) << 52);
  return v * f * f * bits_double((unsigned long long)(1023 + t - 2 * q) << 52);
}
LEM_HD double sums_to_double(long long hi, long long lo, int s) {
  const double v = sums_unscaled(hi, lo);
  bool far = false;
  const double y = scale_near(v, s + 24, &far);
  return far ? scale_far(v, s + 24) : y;
}

}  // namespace oz
}  // namespace lem
