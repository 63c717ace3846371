// Digits, levels and drain schedule of the split-precision GEMM (ozaki.cu):
// how many digits and bits each variant carries, which levels share a pass,
// and at which K steps an accumulator is handed over.  Shared by the kernel's
// issuing thread and its epilogue, which walk the same schedule, and by a host
// check that compiles this header with a plain C++ compiler.
#pragma once

#include <stdint.h>

#ifndef QMLGB_HD
#ifdef __CUDACC__
#define QMLGB_HD __host__ __device__ __forceinline__
#else
#define QMLGB_HD inline
#endif
#endif

#ifdef __CUDACC__
#define QMLGB_UNROLL _Pragma("unroll")
#else
#define QMLGB_UNROLL
#endif

namespace qmlgb {

// S digits of 8 bits, the top one |a_1| <= 2^kTop, kBits = 8 (S - 1) + kTop
// bits in all; levels 2 .. kLMax.  kLow: the levels above 4 exist; the last two then
// share an accumulator, for which digit s carries the weight 2^(-8 (s - 1)).
// kFrac: the output keeps 16 bits below its int64 unit.  kLowBits: the
// low group's unit is level 2's divided by 2^kLowBits.  kStageTiles: digit
// tiles per operand in a ring stage (a K step of the low group, or two K steps
// of three digits).
template <int S>
struct OzDigitsOf;
template <>
struct OzDigitsOf<3> {
  static constexpr int kTop = 8, kBits = 24, kLMax = 4, kLowBits = 0, kStageTiles = 6;
  static constexpr bool kLow = false, kFrac = false;
};
template <>
struct OzDigitsOf<6> {
  static constexpr int kTop = 8, kBits = 48, kLMax = 7, kLowBits = 40, kStageTiles = 6;
  static constexpr bool kLow = true, kFrac = false;
};
template <>
struct OzDigitsOf<7> {
  static constexpr int kTop = 7, kBits = 55, kLMax = 9, kLowBits = 48, kStageTiles = 7;
  static constexpr bool kLow = true, kFrac = true;
};

// Group G of variant S (0: levels 5 and up, 1: levels 2..4).  Its levels are
// its entries 0 .. NE - 1 (the last entry of group 0 holds its last two
// levels), each in one accumulator slot of the four.  The first D are drained:
// entry i after first(i) K steps of a piece and every period(i) from there on,
// never two at one step.  With slots to spare (NE < 4) the entry goes on in the
// one free longest; otherwise it waits for its own.  The others are drained at
// the end of the piece only.
//
// The longest exact chunk, |sum| <= 2^24, from |a_1| <= 2^kTop, |a_s| <= 2^7:
//   kTop = 8: levels 2, 3: 2^16 an element (256 elements, 16 steps), level 4:
//             + 2^14 (204), level 5: + 2^14 (170);
//   kTop = 7: level L: (L - 1) 2^14 (level 4: 341 elements, 5: 256, 6: 204).
// Level 6 of the 48-bit variant, with level 7, runs for 30 steps: a sum past
// 2^24 (digits that all agree in sign) then loses at most 2^2 a product at its
// weight of 2^-48, 2^-47.7 K of the maxima in all, no more than the dropped
// level 8.
// The first hand-overs come late because the epilogue is still writing the
// last tile then (14 us beside 0.8 us a K step; with level 6 drained every 9
// steps from the 4th on, a 6400 x 6400 x 512 update took 0.585 ms), and those
// of one group are spread evenly, since each costs the epilogue about 1000
// clocks (a K step of levels 2..4: 560).
template <int S, int G>
struct OzGroup {
  static constexpr bool kLowGroup = G == 0;
  static constexpr bool kWide = S == 7;
  static constexpr int L0 = kLowGroup ? 5 : 2;
  static constexpr int D = kLowGroup ? 2 : 3;
  static constexpr int NE = kLowGroup ? (kWide ? 4 : 2) : 3;
  static constexpr int NS = 4 - NE;  // slots to spare
  static constexpr bool kSpare = NS > 0;
  static constexpr int kDigits = kLowGroup ? S : 3;
  static constexpr int kSteps = kLowGroup ? 1 : 2;  // K steps per ring stage
  static QMLGB_HD constexpr int first(int i) {
    return kLowGroup ? (kWide ? (i == 0 ? 14 : 12) : (i == 0 ? 10 : 25))
                     : (kWide ? (i == 0 ? 53 : (i == 1 ? 27 : 20)) : 16 - 4 * i);
  }
  static QMLGB_HD constexpr int period(int i) {
    return kLowGroup ? (kWide ? 12 : (i == 0 ? 10 : 30))
                     : (kWide ? (i == 0 ? 60 : (i == 1 ? 30 : 20)) : 12);
  }
  // (first) level of entry i
  static QMLGB_HD constexpr int level(int i) { return L0 + i; }
  // a sum v of entry i adds round(v 2^scale_log) 2^mult_log: the scale undoes
  // the digits' weights; the factor brings level L to the low group's unit, or
  // to 2^shift_top of level 2
  static QMLGB_HD int scale_log(int i) { return OzDigitsOf<S>::kLow ? 8 * (level(i) - 2) : 0; }
  static QMLGB_HD int mult_log(int i, int shift_top) {
    return kLowGroup ? OzDigitsOf<S>::kLowBits - 8 * (level(i) - 2) : shift_top - 8 * i;
  }
};

// Accumulator slots in the order in which they become free, four bits each,
// the first in the lowest: what a piece leaves to the next one.
constexpr uint32_t kOzSlots = 0x3210u;

// The hand-overs of one piece (K steps k0 .. k1) of a group, in order, for the
// issuing thread and the epilogue alike; ord: the slots' order on entry.
template <class Sc>
struct OzHandover {
  int sl[Sc::NE], nb[Sc::D];
  uint32_t spare;  // NS slots, the one free longest in the lowest four bits
  QMLGB_HD OzHandover(int k0, uint32_t ord) : spare(ord >> (4 * Sc::NE)) {
    QMLGB_UNROLL
    for (int i = 0; i < Sc::NE; ++i) sl[i] = (int)(ord >> (4 * i)) & 15;
    QMLGB_UNROLL
    for (int i = 0; i < Sc::D; ++i) nb[i] = k0 + Sc::first(i);
  }
  // the entry handed over at step t, -1 for none
  QMLGB_HD int at(int t) const {
    int e = -1;
    QMLGB_UNROLL
    for (int i = 0; i < Sc::D; ++i) e = t == nb[i] ? i : e;
    return e;
  }
  // the entry handed over next, and its step
  QMLGB_HD int next(int &t) const {
    int e = 0;
    t = nb[0];
    QMLGB_UNROLL
    for (int i = 1; i < Sc::D; ++i)
      if (nb[i] < t) {
        t = nb[i];
        e = i;
      }
    return e;
  }
  QMLGB_HD int slot(int e) const {
    int q = sl[0];
    QMLGB_UNROLL
    for (int i = 1; i < Sc::NE; ++i) q = e == i ? sl[i] : q;
    return q;
  }
  // entry e moves on to the spare slot, or keeps its own
  QMLGB_HD void move(int e) {
    const int old = slot(e);
    QMLGB_UNROLL
    for (int i = 0; i < Sc::D; ++i)
      if (e == i) {
        if (Sc::kSpare) sl[i] = (int)(spare & 15u);
        nb[i] += Sc::period(i);
      }
    if (Sc::kSpare) spare = (spare >> 4) | (uint32_t)old << (4 * (Sc::kSpare ? Sc::NS - 1 : 0));
  }
  // the order after the entries were handed over, 0 .. NE - 1, at the end
  QMLGB_HD uint32_t end() const {
    uint32_t ord = spare;
    QMLGB_UNROLL
    for (int i = 0; i < Sc::NE; ++i) ord |= (uint32_t)sl[i] << (4 * (i + Sc::NS));
    return ord;
  }
};

// Pieces of K (multiples of 4 K steps) over which the undrained sums stay
// below 2^31: kTop = 8 (level 7): 2^17 an element, 960 steps; kTop = 7 (level
// 8 with level 9): 7 2^14 + 2^8, 1152 steps.
QMLGB_HD int oz_pieces(int S, int nk16) {
  const int lim = S == 7 ? 1152 : 960;
  return (nk16 + lim - 1) / lim;
}
QMLGB_HD int oz_piece(int nk16, int nsc, int c) {
  const int n4 = nk16 / 4, q = n4 / nsc, r = n4 % nsc;
  return 4 * (c * q + (c < r ? c : r));
}

// Left shift of level-2 sums in the int64 accumulator: |level-2 sum| <=
// 2^(2 kTop) K, the other levels add less than an eighth of that, so with K
// <= 2^lg the total stays below 2^62.  At least 16 (level 4 is 16 bits below)
// for K <= 2^29 (kTop = 8); 31 is left out: a factor is either below 2^31 (a
// 32-bit multiplier) or a multiple of 2^32 (the upper word alone).
QMLGB_HD int oz_shift_top(int S, int64_t K) {
  int lg = 0;
  while (((int64_t)1 << lg) < K) ++lg;
  const int st = 61 - 2 * (S == 7 ? 7 : 8) - lg;
  return st > 36 ? 36 : (st == 31 ? 30 : st);
}

}  // namespace qmlgb
