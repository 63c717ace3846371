// Host check of csrc/fixconv.cuh's 80-bit and branch-free conversions: acc +
// frac 2^-16 as an exact 128-bit integer, converted by the compiler's
// int128 -> double cast (round to nearest, ties to even) and scaled by a power
// of two, must equal fixed_frac_to_double_bits and normal_double_bits<true>,
// and for frac = 0 normal_double_bits<false>, bit for bit.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <initializer_list>

#include FIXCONV_HEADER

using namespace qmlgb;

static uint64_t s_ = 88172645463325252ull;
static uint64_t rnd() {
  s_ ^= s_ << 13;
  s_ ^= s_ >> 7;
  s_ ^= s_ << 17;
  return s_;
}
static double dbl(uint64_t b) {
  double v;
  std::memcpy(&v, &b, 8);
  return v;
}
static uint64_t bits_of(double v) {
  uint64_t b;
  std::memcpy(&b, &v, 8);
  return b;
}

static int check(int64_t acc, uint32_t frac, int E) {
  const __int128 x = (__int128)acc * 65536 + frac;
  const double ref = std::ldexp((double)x, E - 16);
  for (int neg = 0; neg < 2; ++neg) {
    const uint64_t want = bits_of(neg ? -ref : ref);
    uint64_t got = 0;
    if (!fixed_frac_to_double_bits(acc, frac, E, neg != 0, got) || got != want) {
      std::printf("FAIL frac acc=%lld frac=%u E=%d: %.17g want %.17g\n", (long long)acc, frac, E,
                  dbl(got), dbl(want));
      return 1;
    }
    got = normal_double_bits<true>(acc, frac, E, neg ? 0x80000000u : 0u);
    if (got != want) {
      std::printf("FAIL normal<true> acc=%lld frac=%u E=%d: %.17g want %.17g\n", (long long)acc,
                  frac, E, dbl(got), dbl(want));
      return 1;
    }
    if (frac == 0) {
      got = normal_double_bits<false>(acc, 0, E, neg ? 0x80000000u : 0u);
      if (got != want) {
        std::printf("FAIL normal<false> acc=%lld E=%d\n", (long long)acc, E);
        return 1;
      }
    }
  }
  return 0;
}

int main() {
  const int64_t edge[] = {0, 1, -1, 2, -2, 3, (1ll << 52), (1ll << 53) - 1, (1ll << 53) + 1,
                          -(1ll << 53) - 1, (1ll << 54) + 2, (1ll << 61), -(1ll << 61),
                          (1ll << 62) - 1, -(1ll << 62), (1ll << 47), (1ll << 48) - 1,
                          -(1ll << 48), (1ll << 37) + 1};
  const uint32_t fr[] = {0, 1, 0x7FFF, 0x8000, 0x8001, 0xFFFF, 0x0400, 0x4000};
  for (int64_t a : edge)
    for (uint32_t f : fr)
      for (int E : {-900, -60, 0, 11, 900})
        if (check(a, f, E)) return 1;
  for (int i = 0; i < 2000000; ++i) {
    const int w = 1 + (int)(rnd() % 62);
    int64_t a = (int64_t)(rnd() >> (64 - w));
    if (rnd() & 1) a = -a;
    // exact halves and near-halves of the 53-bit mantissa among them
    if (w > 54 && (rnd() & 3) == 0) a = (a >> (w - 53) << (w - 53)) | (1ll << (w - 54));
    const uint32_t f = (rnd() & 1) ? (uint32_t)(rnd() & 0xFFFF) : fr[rnd() & 7];
    if (check(a, f, (int)(rnd() % 1800) - 900)) return 1;
  }
  std::printf("OK\n");
  return 0;
}
