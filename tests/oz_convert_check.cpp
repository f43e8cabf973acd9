// Host check of the digit arithmetic of the tensor-core FP64 products (oz_convert.h) against
// 128-bit integers: biased_digits against round(x 2^(55 - e)) and the range of every digit,
// sums_to_double against the compiler's conversion of hi 2^24 + lo (round to nearest even)
// scaled by a power of two. Prints "ok <cases>" or the first mismatch and exits 1.
#include <cinttypes>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>

#include "oz_convert.h"

typedef __int128 i128;
static uint64_t rng_state = 0x9E3779B97F4A7C15ull;
static uint64_t next_u64() {  // splitmix64
  uint64_t z = (rng_state += 0x9E3779B97F4A7C15ull);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}
static uint64_t dbits(double d) {
  uint64_t b;
  std::memcpy(&b, &d, 8);
  return b;
}

static void check_digits(uint64_t bits, int e) {
  const int E = lem::oz::exp_field(bits);
  i128 want = 0;
  if (E != 0) {
    const i128 m = i128((bits & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull);
    const int left = E - 1020 - e;  // N = m 2^left
    if (left >= 0)
      want = m << left;
    else if (-left <= 60)
      want = (m + (i128(1) << (-left - 1))) >> -left;
    if (bits >> 63) want = -want;
  }
  const uint64_t N = lem::oz::biased_digits(bits, e);
  i128 sum = 0;
  bool range = (N >> 57) == 0;
  for (int s = 0; s < 7; ++s) {
    const int field = s == 0 ? int((N >> 48) & 0x1FF) : int((N >> (8 * (6 - s))) & 0xFF);
    const int d = field - 128;
    range = range && d >= -128 && d <= 128;
    sum = sum * 256 + d;
  }
  if (sum != want || !range) {
    std::printf("digits of %016" PRIx64 " at scale %d: got %lld, want %lld\n", bits, e, (long long)sum, (long long)want);
    std::exit(1);
  }
}

static void check_sums(long long hi, long long lo, int s) {
  const i128 T = (i128(hi) << 24) + lo;
  const double want = std::ldexp(double(T), s);  // nearest even
  const double got = lem::oz::sums_to_double(hi, lo, s);
  if (dbits(got) != dbits(want)) {
    std::printf("sums %lld %lld 2^%d: got %a, want %a\n", hi, lo, s, got, want);
    std::exit(1);
  }
}

int main(int argc, char** argv) {
  const long long n = argc > 1 ? std::atoll(argv[1]) : 100000;
  long long cases = 0;
  for (int E = 0; E < 2047; ++E)  // every binade under every scale near it
    for (int d = 0; d < 64; ++d) {
      const uint64_t mant[5] = {0, 1, 0xFFFFFFFFFFFFFull, 0x8000000000000ull, next_u64() & 0xFFFFFFFFFFFFFull};
      for (uint64_t m : mant)
        for (uint64_t sign = 0; sign < 2; ++sign, ++cases) check_digits((sign << 63) | (uint64_t(E) << 52) | m, E - 1022 + d);
    }
  for (int sh = 0; sh < 4; ++sh) check_digits(dbits(1.0), 4096), ++cases;
  for (long long i = 0; i < n; ++i) {
    const int a = int(next_u64() % 50) + 1, b = int(next_u64() % 62) + 1;
    long long hi = (long long)(next_u64() >> (64 - a)), lo = (long long)(next_u64() >> (64 - b));
    if (next_u64() & 1) hi = -hi;
    if (next_u64() & 1) lo = -lo;
    if (next_u64() % 8 == 0) hi = 0;
    if (next_u64() % 8 == 0) lo = 0;
    if (next_u64() % 8 == 0) lo = (lo >> 24) << 24;               // exact multiples: ties
    if (next_u64() % 8 == 0) lo = -(hi % (1ll << 20)) * (1 << 24);  // cancellation
    const int s = int(next_u64() % 2200) - 1150;
    check_sums(hi, lo, s);
    check_sums(hi, lo, int(next_u64() % 40) - 1140);
    check_sums(1ll << (a - 1), (long long)((next_u64() & 1) << 23), s);
    check_digits(next_u64() & ~(0x400ull << 52), int(next_u64() % 64) + 1);
    cases += 4;
  }
  std::printf("ok %lld\n", cases);
  return 0;
}
