// Host check of csrc/oz_sched.cuh, the drain schedule of the split-precision
// GEMM: for both groups of every digit count and K from 4 to 1200 steps, the
// accumulator hand-overs of the issuing thread and the reads of the epilogue
// (each replayed as the kernel does it) are the same sequence; the levels
// occupy different slots at all times; and no exact sum can exceed 2^24, nor
// an undrained one 2^31, for the largest digits.
#include <cstdio>
#include <vector>

#include OZ_SCHED_HEADER

using namespace qmlgb;

struct Ev {
  int slot, entry, steps;
};

template <int S, int G>
static double per_element(int L) {
  const double top = (double)(1 << OzDigitsOf<S>::kTop), low = 128.0;
  double m = 0.0;
  for (int s = 1; s <= S; ++s) {
    const int t = L - s;
    if (t < 1 || t > S) continue;
    m += (s == 1 ? top : low) * (t == 1 ? top : low);
  }
  return m;
}

template <int S, int G>
static int check(int k0, int k1, uint32_t &ord_issue, uint32_t &ord_epi) {
  using Sc = OzGroup<S, G>;
  // the issuing thread (issue_piece)
  std::vector<Ev> a, b;
  OzHandover<Sc> H(k0, ord_issue);
  int from[3] = {k0, k0, k0};
  for (int t = k0; t < k1; ++t) {
    int hits = 0;
    for (int i = 0; i < Sc::D; ++i) hits += t == H.nb[i];
    if (hits > 1) return std::printf("FAIL two boundaries S=%d G=%d t=%d\n", S, G, t), 1;
    const int e = H.at(t);
    if (e >= 0) {
      a.push_back({H.slot(e), e, t - from[e]});
      from[e] = t;
      H.move(e);
    }
    // distinct slots, the spare one among them
    unsigned seen = 0;
    for (int i = 0; i < Sc::NS; ++i) seen |= 1u << ((H.spare >> (4 * i)) & 15u);
    for (int i = 0; i < Sc::NE; ++i) seen |= 1u << H.sl[i];
    if (seen != 15u) return std::printf("FAIL slots S=%d G=%d t=%d\n", S, G, t), 1;
  }
  for (int i = 0; i < Sc::NE; ++i) a.push_back({H.sl[i], i, k1 - (i < Sc::D ? from[i] : k0)});
  ord_issue = H.end();
  // the epilogue (drain_piece)
  OzHandover<Sc> E(k0, ord_epi);
  for (int last = 0; last < Sc::NE;) {
    int t;
    int e = E.next(t);
    const bool mid = t < k1;
    if (!mid) e = last++;
    b.push_back({E.slot(e), e, 0});
    if (mid) E.move(e);
  }
  ord_epi = E.end();
  if (ord_issue != ord_epi) return std::printf("FAIL order at the end S=%d G=%d\n", S, G), 1;
  if (a.size() != b.size()) return std::printf("FAIL count S=%d G=%d %d..%d\n", S, G, k0, k1), 1;
  for (size_t i = 0; i < a.size(); ++i) {
    if (a[i].slot != b[i].slot || a[i].entry != b[i].entry || a[i].slot > 3)
      return std::printf("FAIL order S=%d G=%d %d..%d event %zu\n", S, G, k0, k1, i), 1;
    const bool drained = a[i].entry < Sc::D;
    double m = 16.0 * a[i].steps * per_element<S, G>(Sc::level(a[i].entry));
    // the two lowest levels share the last entry of the low group
    if (G == 0 && a[i].entry == Sc::NE - 1)
      m += 16.0 * a[i].steps * per_element<S, G>(Sc::level(a[i].entry) + 1) / 256.0;
    // (level 6 of the 48-bit variant may pass 2^24, see oz_sched.cuh)
    const bool loose = S == 6 && Sc::level(a[i].entry) == 6;
    if (m > (drained ? (loose ? 4.0 : 1.0) * 16777216.0 : 2147483647.0))
      return std::printf("FAIL bound S=%d G=%d level %d steps %d: %g\n", S, G,
                         Sc::level(a[i].entry), a[i].steps, m), 1;
  }
  if (OzDigitsOf<S>::kStageTiles < Sc::kDigits * Sc::kSteps)
    return std::printf("FAIL stage S=%d G=%d\n", S, G), 1;
  return 0;
}

template <int S>
static int all(int lim) {
  int bad = 0;
  for (int nk = 4; nk <= 3 * lim && !bad; nk += nk < 256 ? 4 : 52) {
    const int nsc = oz_pieces(S, nk);
    if (oz_piece(nk, nsc, 0) != 0 || oz_piece(nk, nsc, nsc) != nk)
      return std::printf("FAIL pieces S=%d nk=%d\n", S, nk), 1;
    uint32_t oi = kOzSlots, oe = kOzSlots;
    for (int c = 0; c < nsc && !bad; ++c) {
      const int k0 = oz_piece(nk, nsc, c), k1 = oz_piece(nk, nsc, c + 1);
      if (k1 <= k0 || k0 % 4 || k1 - k0 > lim)
        return std::printf("FAIL piece S=%d nk=%d c=%d: %d..%d\n", S, nk, c, k0, k1), 1;
      if (OzDigitsOf<S>::kLow) bad |= check<S, 0>(k0, k1, oi, oe);
      bad |= check<S, 1>(k0, k1, oi, oe);
    }
  }
  // the int64 total: level 2 alone stays within 2^61, and the shifts exist
  for (int lg = 6; lg < 28 && !bad; ++lg) {
    const int st = oz_shift_top(S, (int64_t)1 << lg);
    if (st < 16 || st > 36 || 2 * OzDigitsOf<S>::kTop + lg + st > 61 ||
        st == 31 || (OzDigitsOf<S>::kLow && OzDigitsOf<S>::kLowBits - st < 1))
      return std::printf("FAIL shift S=%d lg=%d st=%d\n", S, lg, st), 1;
  }
  return bad;
}

int main() {
  if (all<3>(960) || all<6>(960) || all<7>(1152)) return 1;
  std::printf("OK\n");
  return 0;
}
