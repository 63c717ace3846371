// int64 fixed-point -> float64 with integer operations only.
//
// The split-precision product ends with one signed 64-bit fixed-point sum per
// output, to be scaled by a power of two.  Converting it with the float64
// unit costs one float64-pipe instruction per output, and the float64 pipe of
// this part issues about one and a half per clock per SM; with integer
// operations (leading-zero count, shifts, one rounding step) the conversion
// runs on the integer pipes instead.  The result is the IEEE round-to-nearest
// (ties to even) value of acc, as a (double) cast gives, with the exponent
// then moved by E.  The body compiles as CUDA device code and as plain C++
// (the host test checks it against the cast).
#pragma once

#include <stdint.h>

#if defined(__CUDACC__)
#define QMLGB_HD __host__ __device__ __forceinline__
#else
#define QMLGB_HD inline
#endif

namespace qmlgb {

QMLGB_HD int clz64(uint64_t x) {
#if defined(__CUDA_ARCH__)
  return __clzll((long long)x);
#else
  return __builtin_clzll(x);
#endif
}

// Bit pattern of round(acc) 2^E (round to nearest, ties to even), sign
// flipped when neg.  False when the result would not be a normal float64 (the
// caller then scales another way); acc = 0 gives a signed zero.
QMLGB_HD bool fixed_to_double_bits(int64_t acc, int E, bool neg, uint64_t &bits) {
  const uint64_t flip = neg ? 0x8000000000000000ull : 0ull;
  if (acc == 0) {
    bits = flip;
    return true;
  }
  const uint64_t sgn = acc < 0 ? 0x8000000000000000ull : 0ull;
  const uint64_t u = acc < 0 ? (uint64_t)0 - (uint64_t)acc : (uint64_t)acc;
  const int lz = clz64(u);
  const uint64_t m = u << lz;   // leading one at bit 63
  uint64_t mant = m >> 11;      // 53 significant bits
  const uint64_t rem = m & 0x7FFull;
  int e2 = 63 - lz;             // u lies in [2^e2, 2^(e2 + 1))
  if (rem > 0x400ull || (rem == 0x400ull && (mant & 1ull))) {
    ++mant;
    if (mant >> 53) {  // rounded up to the next power of two
      mant >>= 1;
      ++e2;
    }
  }
  const int bexp = e2 + 1023 + E;
  if (bexp <= 0 || bexp >= 2047) return false;
  bits = (sgn ^ flip) | ((uint64_t)bexp << 52) | (mant & 0xFFFFFFFFFFFFFull);
  return true;
}

// The same for acc + frac 2^-16 (frac < 2^16): an 80-bit fixed-point number,
// brought to 64 significant bits (what falls below rounds the value only as a
// sticky bit) and rounded once.
QMLGB_HD bool fixed_frac_to_double_bits(int64_t acc, uint32_t frac, int E, bool neg,
                                        uint64_t &bits) {
  const bool below = acc < 0;
  uint64_t hi = below ? ~(uint64_t)acc + (frac == 0 ? 1u : 0u) : (uint64_t)acc;
  const uint32_t lo = below && frac ? 0x10000u - frac : frac;
  const int lz = hi ? clz64(hi) : 64;
  const int s = lz < 17 ? (lz > 1 ? lz - 1 : 0) : 16;  // keep the sign bit clear
  const uint64_t rest = (uint64_t)lo & ((1ull << (16 - s)) - 1ull);
  uint64_t u = (hi << s) | ((uint64_t)lo >> (16 - s));
  if (rest) u |= 1ull;  // only when u has at least 62 significant bits
  const int64_t v = below ? -(int64_t)u : (int64_t)u;
  return fixed_to_double_bits(v, E - s, neg, bits);
}

// The same two conversions, without branches, for an E that keeps every result
// normal or zero (-980 < E < 940): a zero sum gives +0 (or -0 with flip).  The
// implicit bit of the mantissa carries into the exponent field, which is
// therefore one less, and so does a rounding up to the next power of two.
// flip: 0x80000000 to negate, else 0.
template <bool FRAC>
QMLGB_HD uint64_t normal_double_bits(int64_t acc, uint32_t frac, int E, uint32_t flip) {
  const uint64_t neg = (uint64_t)(acc >> 63);  // all ones when below zero
  uint64_t u = ((uint64_t)acc ^ neg) - neg;
  int lz;
  uint64_t m;
  if (FRAC) {
    // 80 bits: u less one and frac's complement when below zero with a fraction
    const uint32_t lo = neg && frac ? 0x10000u - frac : frac;
    u -= neg && frac ? 1u : 0u;
    lz = u ? clz64(u) : 64;
    // shift by up to 16 places, bits of lo coming in (the sticky bit cannot
    // matter unless u fills 48 bits and more, where it lies below the rounding
    // bit of a 53-bit mantissa only when lz < 11: kept there)
    const int s = lz < 16 ? lz : 16;
    const uint64_t rest = (uint64_t)lo & ((1ull << (16 - s)) - 1ull);
    u = (u << s) | ((uint64_t)lo >> (16 - s)) | (rest ? 1u : 0u);
    lz = u ? clz64(u) : 63;
    m = u << lz;
    E -= s;
  } else {
    lz = clz64(u | 1u);
    m = u << lz;
  }
  uint64_t mant = ((m >> 10) + 1u) >> 1;                 // half up
  mant &= ~(uint64_t)((m & 0x7FFull) == 0x400ull);       // ties to even
  uint64_t bits = mant + ((uint64_t)(uint32_t)(63 - lz + 1022 + E) << 52);
  bits |= neg & 0x8000000000000000ull;
  if (m == 0) bits = 0;
  return bits ^ ((uint64_t)flip << 32);
}

}  // namespace qmlgb
