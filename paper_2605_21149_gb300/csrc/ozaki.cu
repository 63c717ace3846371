// Split-precision float64 GEMM on tcgen05 tensor cores (Ozaki-style).
//
//   C <- alpha op(A) op(B) + beta C,  op(A) m x K, op(B) K x n, float64 in/out.
//
// Each row i of op(A) is scaled by 2^-e_i (|x| <= 2^e_i), rounded to an integer
// of 8 (S - 1) + T bits and written as S signed digits of 8 bits, |a_1| <= 2^T
// and |a_s| <= 2^7 (s >= 2), every digit an integer that bf16 holds exactly;
// the same for the columns of op(B) with exponents f_j.  With level L = s + t,
//   C_ij = 2^(e_i+f_j-2T) sum_{L <= LMAX} 2^(-8(L-2)) sum_{s+t=L} (A_s B_t^T)_ij
// (products below the truncation level are dropped).  Two digit counts carry
// the library's precisions:
//   S = 6 (T = 8, levels 2..7): 48 bits, 21 digit products -- QML_SPLIT_BF16;
//   S = 7 (T = 7, levels 2..9): 55 bits, 34 digit products -- the large
//       contractions of QML_FP64: an operand's rounding (2^-56 of its row's
//       maximum) and the dropped levels (about 2^-58 sqrt(K) of the maxima's
//       product) lie below the rounding of a float64 accumulation;
// and S = 3 (levels 2..4) serves callers that ask for 24 bits or fewer.  All
// products of one level carry the same weight and are integers, so they add
// up exactly in an FP32 TMEM accumulator as long as the sum stays below 2^24:
// whatever the tensor core's order or rounding.  Levels 2..6, whose last bits
// matter, are therefore read out ("drained") every chunk of K that cannot
// exceed that bound (oz_sched.cuh); the levels below (S = 6: 7, in level 6's
// accumulator; S = 7: 7, and 8 with 9 in one accumulator) carry weights of 2^-40
// and less, where FP32 rounding costs less than the dropped levels.
// Why 8-bit digits: 6-bit digits allow chunks of 1536 elements but need 36
// products for 48 bits; 8-bit digits need 21 and pay for it with a drain
// every 160..512 elements, which the epilogue warps do beside the MMAs.
//
// Fixed point.  A drained sum is converted to int32 and added, times a power
// of two, into one int64 accumulator per output (one multiply-add).  The low
// levels come first, exactly, in units of the lowest level; they are then
// shifted to the final unit 2^-shift_top of level 2 (S = 7 keeps the 16 bits
// below it in half a register), and the high levels added.  One conversion to
// float64 per output, by integer operations (fixconv.cuh); the scaling by a
// power of two is an integer add to the exponent field, and the digit slicing
// reads the float64 bit patterns with integer operations (the float64 pipe of
// this part is narrow).  A row that holds an infinity or a NaN has the
// exponent kNanExp and no digits; every output it takes part in is NaN.
//
// Groups.  The levels are taken in two groups, low first: {5 ..} in one pass
// over K with all S digits, then {2, 3, 4} with three.  Every K step of 16
// loads each digit tile the group needs once and runs all of its products.
// TMEM holds four 128-column accumulators (slots).  Drained levels change
// slots at their chunk boundaries, which are staggered; with a slot to spare
// (S = 6: two in the first group, one in the second; S = 7: one in the second)
// the next chunk starts at once, and without one the other levels' products of that K step go
// first and cover the drain.  A group takes over the slots in the order in
// which the one before it leaves them, each when its first product needs it.
// What bounds a K step is the rate at which the issuing warp hands MMAs over:
// 71 clocks each with operands in uniform registers (93 from a one-lane branch;
// cuBLAS's 1900 TFLOP/s would be 87 at the burst clock, 64 the tensor core's
// own rate).  A pair of CTAs on M = 256 MMAs (cta_group::2, half the B traffic in
// shared memory) ran no faster, 99, and clusters of two that shared B's digit
// tiles by multicast no faster than single CTAs in bands: 16000^2 K = 512 2.56
// against 1.86 ms, W = X^T X of 6900 x 5952 3.5-3.8 against 3.5-3.8, TQU Nside 16
// solve (QML_FP64) 38.4 against 37.9, QU Nside 32 295.4 against 292.8.
//
// Digit layout.  The slicing kernel writes the digits in the order and the
// shared-memory image the MMA wants: [128-row tile][K step][digit] tiles of
// 4 KB (128 rows x 16 elements, 32-byte swizzle).  What a K step needs of an
// operand, digits 1..d, is one contiguous run, fetched by one linear bulk
// copy; 32-byte rows through tensor maps had been what bounded the product.
//
// Kernel layout: one CTA per 128 x 128 output tile (128 x 64 where those fit
// one wave), 384 threads.
//   warp 0   producer (one lane): bulk copies into a ring of stages, guarded
//            by mbarriers;
//   warp 1   TMEM allocator and MMA issuer (in step, one lane issuing): tcgen05.mma kind::f16
//            M=128 N=128 (64) K=16; commits a slot to the epilogue at the end of a
//            chunk and waits for it to be read before refilling it;
//   warps 2-3 idle (they complete warpgroup 0 for the register split);
//   warps 4-11 epilogue: warp w reads TMEM lanes 32 (w % 4) .. +31 (tile rows)
//            and 64 columns (half (w - 4) / 4 of the tile) of each slot.
// Every mbarrier wait is bounded (2 s of %globaltimer): on expiry the CTA records
// QML_ETIMEOUT, drains what it issued, frees TMEM and returns.
#include "fixconv.cuh"
#include "oz_order.cuh"
#include "oz_sched.cuh"
#include "internal.cuh"
#include "ptx.cuh"

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <mutex>

namespace qmlgb {

namespace {

constexpr int OBM = 128, OBN = 128, OBK = 64;  // output tile; K padding of the digits
constexpr int KS = 16;                          // K per MMA instruction
constexpr int kDigitTile = OBM * KS * 2;        // 4 KB: one 128 x 16 bf16 digit tile
// Three warpgroups.  Warpgroup 0: warp 0 the producer, warp 1 the TMEM
// allocator and MMA issuer, warps 2-3 idle.  Warpgroups 1 and 2 (warps
// 4-11): kEpiWarps epilogue warps, each one TMEM lane quarter (32 tile rows)
// by half of the tile's columns, so a thread holds 64 int64 accumulators.  The
// block starts at kLaunchRegs registers a thread (12 warps, three on each SM
// sub-partition of 16384 registers: 65536 / 384 rounded down to 8); then
// warpgroup 0 gives registers back (setmaxnreg.dec to kIssueRegs) and the
// epilogue takes them (setmaxnreg.inc to kEpiRegs), so that its 64 int64 sums
// stay in registers.  The split adds up exactly:
// 128 kIssueRegs + 256 kEpiRegs = 384 kLaunchRegs.
constexpr int kEpiWarps = 8;
constexpr int kThreads = 128 + 32 * kEpiWarps;
constexpr int kLaunchRegs = 168, kIssueRegs = 56, kEpiRegs = 224;
static_assert(128 * kIssueRegs + 256 * kEpiRegs == kThreads * kLaunchRegs,
              "register split must equal the launch's registers");
static_assert(kThreads * kLaunchRegs <= 65536, "launch registers exceed the SM");

// ------------------------------------------------------------ PTX helpers --
// (bulk copy, tcgen05 and shared-memory descriptor helpers: ptx.cuh)

// instruction descriptor, kind::f16: D f32, A and B bf16, both K-major, N, M
template <int NT>
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(NT >> 3) << 17) |
                            ((uint32_t)(OBM >> 4) << 24);
// Tile widths.  NT = 128 is the general form.  NT = kNarrow halves a tile (one
// CTA per 128 x 64, B's digit tiles fetched by halves): a product of up to half
// as many 128-wide tiles as there are SMs takes one tile's time whatever its
// size, MMAs and output both in proportion to the width.
constexpr int kNarrow = 64;

// K-major bf16 tile of 16-element (32-byte) rows with the 32-byte swizzle
// (8-row atoms of 256 B): start address, LBO 16 B (unused: one MMA's K is the
// whole swizzle row), SBO 256 B, descriptor version 1, layout type 6.
__device__ __forceinline__ uint64_t smem_desc_sw32(uint32_t saddr) {
  uint64_t d = (uint64_t)((saddr >> 4) & 0x3FFFu);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(256 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)6 << 61;
  return d;
}

// S = 7 keeps the low halves of its sums in shared memory between the groups
// (in registers they pushed the epilogue into spills: 64 int64 sums and the
// loaded columns fill the 168 the compiler allots)
template <int S>
constexpr int kResidBytes = OzDigitsOf<S>::kFrac ? 32 * 32 * kEpiWarps * 4 : 0;

// 1.5 2^23 as a float and its bit pattern
constexpr float kMagicF = 12582912.0f;
constexpr uint32_t kMagicI = 0x4B400000u;

struct OzParams {
  int64_t M, N;            // logical output size
  const unsigned char *DA, *DB;  // digit tiles of op(A), op(B)^T (first row tile)
  int nk16;                // K steps of 16
  int nstages;             // ring depth
  int nsc;                 // pieces of K whose undrained sums fit an int32
  int shift_top;           // left shift of level-2 sums in the int64 accumulator
  int tiles_m, tiles_n, lower;
  int band;                // tile rows per band of the work order (>= 1)
  int ntiles;              // work items, taken round-robin by the grid
  double alpha, betac;
  int alpha_pow2, alpha_exp, alpha_neg;  // alpha = (-1)^neg 2^exp when alpha_pow2
  // 0: C is not read (beta = 0); 1: v + C (beta = 1); 2: fma(beta, C, v).  A
  // float64 compare is a float64-pipe instruction (tens of clocks a warp on
  // this part), so the output takes this integer instead of testing beta.
  int beta_mode;
  int prefetch_c;  // fetch each output tile's C into L2 when the tile starts
  double *C;
  int64_t ldc;
  const int *ea, *eb;
  DevStatus *status;
  // failure-path test (tuning key test_wait_timeout): the producer issues no
  // copies and every wait gives up after wait_ns, so each CTA takes its
  // timeout exit; normal calls have wait_ns = kWaitNs and no_loads = 0
  uint64_t wait_ns;
  int no_loads;
};

// The output tile of work item `item` (NT < 128: a part of one) and the part's
// first column, which lies past the last one for some parts: every role of a
// CTA passes over those.
template <int NT>
__device__ __forceinline__ void item_tile(const OzParams &p, int item, int &tm, int &tn, int &n0) {
  constexpr int kParts = OBN / NT;
  if (NT == OBN)
    oz_band_tile_of(p.tiles_m, p.tiles_n, p.lower, p.band, item, tm, tn);
  else
    oz_tile_of(p.lower, p.tiles_n, item / kParts, tm, tn);
  n0 = tn * OBN + item % kParts * NT;
}

// Every digit product of level L for one K step: pair (s, L - s) reads digit
// tile s - 1 of A and L - s - 1 of B, at descriptor offsets of 256 (4 KB >> 4;
// 2 NT for B's NT rows) per tile from the step's first tiles (da, db).  Unrolled at compile time,
// so the issuing warp spends a few instructions per MMA: with loop bounds,
// flags and descriptors computed at run time, or moved to uniform registers
// for every MMA, it could not keep up with the tensor core (93 clocks of issue
// per 64-clock MMA; 71 as it is).  The first pair
// writes the accumulator when acc0 is 0 (first K step of a chunk).
template <int S, int L, int NT>
__device__ __forceinline__ void issue_level(uint32_t tmem, uint64_t da, uint64_t db, uint32_t acc0,
                                            uint32_t lead) {
  constexpr int s0 = L - S > 1 ? L - S : 1, s1 = L - 1 < S ? L - 1 : S;
#pragma unroll
  for (int s = s0; s <= s1; ++s)
    mma_bf16_warp(tmem, da + (uint64_t)(256 * (s - 1)), db + (uint64_t)(2 * NT * (L - s - 1)),
                  kIdesc<NT>, s == s0 ? acc0 : 1u, lead);
}

// Output of 8 consecutive columns of one row, general form: C[gi + gj ldc] =
// alpha 2^(e) acc + beta C for the live entries (gj < N, and gj <= gi for a
// lower C), any alpha and beta, results outside the normal range, rows with
// an infinity or a NaN.  Not inlined (rare, and large).  FRAC: r holds, two to
// a word, the 16 bits below each sum's unit.
template <bool FRAC>
__device__ __noinline__ void store_out8(const OzParams &p, int64_t gi, int64_t gj0, int ebase,
                                        long long a0, long long a1, long long a2, long long a3,
                                        long long a4, long long a5, long long a6, long long a7,
                                        uint32_t r0, uint32_t r1, uint32_t r2, uint32_t r3,
                                        int f0, int f1, int f2, int f3, int f4, int f5, int f6,
                                        int f7) {
  const long long av[8] = {a0, a1, a2, a3, a4, a5, a6, a7};
  const uint32_t rv[4] = {r0, r1, r2, r3};
  const int fv[8] = {f0, f1, f2, f3, f4, f5, f6, f7};
  const int eshift = p.alpha_pow2 ? p.alpha_exp : 0;
  const bool aneg = p.alpha_pow2 && p.alpha_neg;
  const int bmode = p.beta_mode;
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const int64_t gj = gj0 + u;
    if (gj >= p.N || (p.lower && gi < gj)) continue;
    const int E = ebase + fv[u];
    const uint32_t fr = FRAC ? (u & 1 ? rv[u >> 1] >> 16 : rv[u >> 1] & 0xFFFFu) : 0u;
    uint64_t bits;
    double v;
    if (E > kNanExp / 2) {  // a row with an infinity or a NaN
      v = __longlong_as_double(0x7FF8000000000000ll);
    } else if (FRAC ? fixed_frac_to_double_bits(av[u], fr, E + eshift, aneg, bits)
                    : fixed_to_double_bits(av[u], E + eshift, aneg, bits)) {
      v = __longlong_as_double((long long)bits);
      if (!p.alpha_pow2) v *= p.alpha;
    } else {
      v = p.alpha * ldexp((double)av[u] + (double)fr * (1.0 / 65536.0), E);
    }
    if (bmode == 1) v += p.C[gi + gj * p.ldc];
    else if (bmode == 2) v = fma(p.betac, p.C[gi + gj * p.ldc], v);
    p.C[gi + gj * p.ldc] = v;
  }
}

// The common output: alpha = +-2^k, beta 0 or 1 (ADD), every result a normal
// float64 or zero.  A float64 instruction holds its SM sub-partition about 76
// clocks a warp on this part, and one that the compiler predicates off or
// selects away costs the same; the general form above spent 25 us of a tile's
// time on them (K = 512 trailing update of 6400: 0.76 ms, 0.46 without any
// output).  Here the conversion is integer throughout (normal_double_bits)
// and beta = 1 costs the one addition it needs.
// Columns 8 g .. 8 g + 7: c points at the first, lim is the number of live
// columns from there on; fNM: two column exponents, 16 bits each; c0 .. c7: the
// entries of C for ADD, read by the caller a group ahead.  Not inlined: the 8
// calls of a tile share one copy of the code (about 45 instructions an output;
// 64 copies of it did not stay in the instruction cache).
template <bool FRAC, bool ADD>
__device__ __noinline__ void store_fast8(double *c, int64_t ldc, int lim, int E0, uint32_t sflip,
                                         long long a0, long long a1, long long a2, long long a3,
                                         long long a4, long long a5, long long a6, long long a7,
                                         uint32_t r0, uint32_t r1, uint32_t r2, uint32_t r3,
                                         uint32_t f01, uint32_t f23, uint32_t f45, uint32_t f67,
                                         double c0, double c1, double c2, double c3, double c4,
                                         double c5, double c6, double c7) {
  const long long av[8] = {a0, a1, a2, a3, a4, a5, a6, a7};
  const uint32_t rv[4] = {r0, r1, r2, r3};
  const uint32_t fv[4] = {f01, f23, f45, f67};
  const double cv[8] = {c0, c1, c2, c3, c4, c5, c6, c7};
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const uint32_t fr = FRAC ? (u & 1 ? rv[u >> 1] >> 16 : rv[u >> 1] & 0xFFFFu) : 0u;
    const int f = u & 1 ? (int)fv[u >> 1] >> 16 : (int)(short)fv[u >> 1];
    const uint64_t bits = normal_double_bits<FRAC>(av[u], fr, E0 + f, sflip);
    double v = __longlong_as_double((long long)bits);
    if (ADD) v += cv[u];
    if (u < lim) c[u * ldc] = v;
  }
}

// One piece (K steps k0 .. k1) of group G on the issuing thread; see
// oz_sched.cuh for the schedule it shares with the epilogue.
struct Issuer {
  uint32_t tbase, full0, empty0, accf, acce, smem0;
  int stage_bytes, nst;
  DevStatus *st;
  uint64_t wait_ns;
  int stage;
  uint32_t phase;
  uint32_t used, par;  // per slot: filled before; parity of the drain to wait for
  uint32_t ord;        // slots in the order in which they become free
  uint32_t lead;       // set in the lane that issues
};
// (every lane waits, and all go on or none)
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, const Issuer &I) {
  return __all_sync(0xffffffffu, mbar_wait(bar, parity, I.st, I.wait_ns)) != 0;
}
template <int N>
struct IntC {
  static constexpr int value = N;
};

__device__ __forceinline__ bool slot_acquire(Issuer &I, int q) {
  if ((I.used >> q) & 1) {
    if (!warp_wait(I.acce + 8 * q, (I.par >> q) & 1, I)) return false;
    I.par ^= 1u << q;
    tc_fence_after();
  }
  I.used |= 1u << q;
  return true;
}

// the products of entry E of group G for one K step
template <int S, int G, int E, int NT>
__device__ __forceinline__ void issue_entry(uint32_t tmem, uint64_t da, uint64_t db, uint32_t acc0,
                                            uint32_t lead) {
  using Sc = OzGroup<S, G>;
  if constexpr (E < Sc::NE) {
    issue_level<S, Sc::L0 + E, NT>(tmem, da, db, acc0, lead);
    if constexpr (Sc::kLowGroup && E == Sc::NE - 1)
      issue_level<S, Sc::L0 + E + 1, NT>(tmem, da, db, 1u, lead);
  }
}

template <int S, int NT, int G>
__device__ __forceinline__ bool issue_piece(Issuer &I, int k0, int k1) {
  using Sc = OzGroup<S, G>;
  OzHandover<Sc> H(k0, I.ord);
  for (int ks = k0; ks < k1; ks += Sc::kSteps) {
    if (!warp_wait(I.full0 + 8 * I.stage, I.phase, I)) return false;
    tc_fence_after();
    const uint32_t sa = I.smem0 + (uint32_t)(I.stage * I.stage_bytes);
    const uint64_t da0 = smem_desc_sw32(sa), db0 = smem_desc_sw32(sa + (uint32_t)(I.stage_bytes >> 1));
#pragma unroll
    for (int j = 0; j < Sc::kSteps; ++j) {
      const uint64_t da = da0 + (uint64_t)(256 * Sc::kDigits * j);
      const uint64_t db = db0 + (uint64_t)(2 * NT * Sc::kDigits * j);
      const int t = ks + j;
      // entry bl starts its next chunk here: its slot goes to the epilogue now,
      // and with a spare slot the entry goes on in that one; without, the other
      // entries go first and cover the wait
      const int bl = H.at(t);
      if (bl >= 0) {
        mma_commit_warp(I.accf + 8 * H.slot(bl), I.lead);
        H.move(bl);
      }
      // a slot is waited for just before its first product
      auto entry = [&](auto E) -> bool {
        constexpr int e = decltype(E)::value;
        if (e >= Sc::NE) return true;
        if (!Sc::kSpare && bl == e) return true;
        const bool fresh = t == k0 || bl == e;
        const int q = H.sl[e < Sc::NE ? e : 0];
        if (fresh && !slot_acquire(I, q)) return false;
        issue_entry<S, G, e, NT>(I.tbase + 128 * q, da, db, fresh ? 0u : 1u, I.lead);
        return true;
      };
      if (!entry(IntC<0>{}) || !entry(IntC<1>{}) || !entry(IntC<2>{}) || !entry(IntC<3>{}))
        return false;
      if (!Sc::kSpare && bl >= 0) {
        const int q = H.slot(bl);
        if (!slot_acquire(I, q)) return false;
        if (bl == 0)
          issue_entry<S, G, 0, NT>(I.tbase + 128 * q, da, db, 0u, I.lead);
        else
          issue_entry<S, G, 1, NT>(I.tbase + 128 * q, da, db, 0u, I.lead);
      }
    }
    // frees the smem slot when these MMAs finish
    mma_commit_warp(I.empty0 + 8 * I.stage, I.lead);
    if (++I.stage == I.nst) {
      I.stage = 0;
      I.phase ^= 1;
    }
  }
#pragma unroll
  for (int i = 0; i < Sc::NE; ++i) mma_commit_warp(I.accf + 8 * H.sl[i], I.lead);
  I.ord = H.end();
  return true;
}

// The producer's loads of one piece of group G: a stage holds kSteps K steps
// of kDigits digit tiles per operand; one bulk copy per operand and K step.
struct Producer {
  uint32_t full0, empty0, smem0;
  int stage_bytes, nst;
  DevStatus *st;
  uint64_t wait_ns;
  int stage;
  uint32_t phase;
  int last_phase[4];
};

template <int S, int NT, int G>
__device__ __forceinline__ bool load_piece(Producer &P, const unsigned char *a,
                                           const unsigned char *b, int k0, int k1) {
  using Sc = OzGroup<S, G>;
  constexpr uint32_t kRun = Sc::kDigits * kDigitTile;
  for (int ks = k0; ks < k1; ks += Sc::kSteps) {
    if (!mbar_wait(P.empty0 + 8 * P.stage, P.phase ^ 1, P.st, P.wait_ns)) return false;
    const uint32_t fb = P.full0 + 8 * P.stage;
    mbar_expect_tx(fb, Sc::kSteps * (kRun + kRun / OBN * NT));
    const uint32_t sa = P.smem0 + (uint32_t)(P.stage * P.stage_bytes);
    const uint32_t sb = sa + (uint32_t)(P.stage_bytes >> 1);
#pragma unroll
    for (int j = 0; j < Sc::kSteps; ++j) {
      const size_t src = (size_t)(ks + j) * S * kDigitTile;
      bulk_load(sa + j * kRun, a + src, kRun, fb);
      if constexpr (NT < OBN) {
        // this tile's rows of each of B's digit tiles
        constexpr uint32_t kPart = kDigitTile / OBN * NT;
#pragma unroll
        for (int q = 0; q < Sc::kDigits; ++q)
          bulk_load(sb + (j * Sc::kDigits + q) * kPart, b + src + q * kDigitTile, kPart, fb);
      } else {
        bulk_load(sb + j * kRun, b + src, kRun, fb);
      }
    }
    P.last_phase[P.stage] = (int)P.phase;
    if (++P.stage == P.nst) {
      P.stage = 0;
      P.phase ^= 1;
    }
  }
  return true;
}

// S: digit count (OzGroup); persistent: each CTA takes the work items
// blockIdx.x, + gridDim.x, ...; the producer runs on into the next tile's data and the
// MMAs of the next tile start as soon as the epilogue has read the
// accumulators, while the epilogue converts and stores the finished tile from
// its registers.
template <int S, int NT>
__global__ void __launch_bounds__(kThreads, 1) ozaki_gemm_kernel(const __grid_constant__ OzParams p) {
  constexpr int kEpiCols = NT * 4 / kEpiWarps;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  // 1024-byte alignment for the swizzled tiles
  unsigned char *smem = (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const int NST = p.nstages;
  constexpr int stage_bytes = 2 * OzDigitsOf<S>::kStageTiles * kDigitTile;  // A tiles, then B tiles
  // S = 7: the 16 bits below each sum's unit, two to a word, [pair][thread]
  uint32_t *resid = (uint32_t *)(smem + (size_t)NST * stage_bytes);
  uint64_t *bars = (uint64_t *)((unsigned char *)resid + kResidBytes<S>);
  // bars: [0,NST) full, [NST,2NST) empty, then 4 slots filled, 4 slots read, drain
  uint32_t *tmem_holder = (uint32_t *)(bars + 2 * NST + 9);

  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  DevStatus *st = p.status;
  const uint32_t full0 = smem_u32(&bars[0]), empty0 = smem_u32(&bars[NST]);
  const uint32_t accf = smem_u32(&bars[2 * NST]), acce = smem_u32(&bars[2 * NST + 4]);
  const uint32_t drain = smem_u32(&bars[2 * NST + 8]);

  if (threadIdx.x == 0) {
    for (int s = 0; s < NST; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    for (int q = 0; q < 4; ++q) {
      mbar_init(accf + 8 * q, 1);
      mbar_init(acce + 8 * q, kEpiWarps);
    }
    mbar_init(drain, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) tmem_alloc(smem_u32(tmem_holder), 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tbase = __shfl_sync(0xffffffffu, *tmem_holder, 0);

  if (warp < 4) {
  // warpgroup 0 hands registers to the epilogue warpgroups
  if constexpr (NT == OBN) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kIssueRegs));
  if (warp == 0) {
    // ----------------------------------------------------------- producer
    if (lane == 0) {
      Producer P{full0, empty0, smem_u32(smem), stage_bytes, NST, st, p.wait_ns, 0, 0,
                 {-1, -1, -1, -1}};
      bool ok = (*((volatile int *)&st->code) == 0) && !p.no_loads;
      for (int item = blockIdx.x; item < p.ntiles && ok; item += gridDim.x) {
        int tm, tn, n0;
        item_tile<NT>(p, item, tm, tn, n0);
        if (NT < OBN && n0 >= p.N) continue;
        const size_t rt_bytes = (size_t)p.nk16 * S * kDigitTile;
        const unsigned char *a = p.DA + (size_t)tm * rt_bytes;
        const unsigned char *b =
            p.DB + (size_t)tn * rt_bytes + (size_t)(n0 - tn * OBN) * (KS * 2);
        if constexpr (OzDigitsOf<S>::kLow)
          for (int c = 0; c < p.nsc && ok; ++c)
            ok = load_piece<S, NT, 0>(P, a, b, oz_piece(p.nk16, p.nsc, c),
                                      oz_piece(p.nk16, p.nsc, c + 1));
        for (int c = 0; c < p.nsc && ok; ++c)
          ok = load_piece<S, NT, 1>(P, a, b, oz_piece(p.nk16, p.nsc, c),
                                    oz_piece(p.nk16, p.nsc, c + 1));
      }
      if (!ok) {
        // drain: wait (bounded) until the last load issued into each slot has
        // landed, so no copy is still writing shared memory when the CTA exits
        for (int q = 0; q < NST; ++q)
          if (P.last_phase[q] >= 0) mbar_drain_wait(full0 + 8 * q, (uint32_t)P.last_phase[q]);
      }
    }
  } else if (warp == 1) {
    // -------------------------------------------------------- MMA issuer
    // (the whole warp in step, one lane issuing)
    {
      Issuer I{tbase, full0, empty0, accf, acce, smem_u32(smem), stage_bytes, NST, st, p.wait_ns,
               0, 0, 0, 0, kOzSlots, elect_lane()};
      bool ok = __all_sync(0xffffffffu, *((volatile int *)&st->code) == 0) != 0;
      for (int item = blockIdx.x; item < p.ntiles && ok; item += gridDim.x) {
        if constexpr (NT < OBN) {
          int tm, tn, n0;
          item_tile<NT>(p, item, tm, tn, n0);
          if (n0 >= p.N) continue;
        }
        if constexpr (OzDigitsOf<S>::kLow)
          for (int c = 0; c < p.nsc && ok; ++c)
            ok = issue_piece<S, NT, 0>(I, oz_piece(p.nk16, p.nsc, c),
                                       oz_piece(p.nk16, p.nsc, c + 1));
        for (int c = 0; c < p.nsc && ok; ++c)
          ok = issue_piece<S, NT, 1>(I, oz_piece(p.nk16, p.nsc, c),
                                     oz_piece(p.nk16, p.nsc, c + 1));
      }
      // wait for every MMA this thread issued before TMEM is released
      mma_commit_warp(drain, I.lead);
      mbar_drain_wait(drain, 0);
    }
  }
  } else {
    if constexpr (NT == OBN) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kEpiRegs));
    // ---------------------------------------------------------- epilogue
    const int quad = warp & 3;            // TMEM lane quarter this warp may access
    const int half = (warp - 4) >> 2;     // which kEpiCols columns of the tile
    const int row = quad * 32 + lane;
    const uint32_t lane_base = tbase + ((uint32_t)(quad * 32) << 16) + kEpiCols * half;
    constexpr bool FRAC = OzDigitsOf<S>::kFrac;
    uint32_t par = 0;  // per slot: parity of the fill to wait for
    uint32_t ord = kOzSlots;
    bool ok = true;
    long long acc[kEpiCols];
    uint32_t *res = resid + (threadIdx.x - 128);  // stride 32 kEpiWarps
    long long bias = 0;
    // Reads slot q: acc += round(sum 2^scale_log) 2^mult_log.  The float to
    // integer conversion is an addition of 1.5 2^23, exact below 2^22 and
    // checked for every value (F2I issues an eighth as fast); the constant in
    // its bit pattern is collected in `bias` and taken off with the shift.
    auto drain_slot = [&](int q, int scale_log, int mult_log) -> bool {
      int okw = 1;
      if (lane == 0) okw = mbar_wait(accf + 8 * q, (par >> q) & 1, st, p.wait_ns) ? 1 : 0;
      par ^= 1u << q;
      okw = __shfl_sync(0xffffffffu, okw, 0);
      __syncwarp();
      if (!okw) return false;
      tc_fence_after();
      const uint32_t lbase = lane_base + 128 * q;
      const float scale = __int_as_float((127 + scale_log) << 23);
      const bool high = mult_log >= 32;  // only the upper word changes
      constexpr int kLd = 32;  // columns in flight that the registers hold
      const int mult = 1 << (high ? mult_log - 32 : mult_log);
#pragma unroll
      for (int cb = 0; cb < kEpiCols / kLd; ++cb) {
        uint32_t a[kLd];
        auto load = [&] {
          tmem_ld32_async(lbase + kLd * cb, a);
          tmem_ld_wait();
          // (the loaded registers pass through the wait, so no use moves above it)
#pragma unroll
          for (int j = 0; j < kLd; ++j) asm volatile("" : "+r"(a[j]));
        };
        load();
        uint32_t off = 0;
#pragma unroll
        for (int j = 0; j < kLd; ++j) {
          a[j] = __float_as_uint(fmaf(__uint_as_float(a[j]), scale, kMagicF));
          off |= a[j] ^ kMagicI;
        }
        if (__any_sync(0xffffffffu, (off >> 23) != 0)) {
          // a sum past 2^22 in some lane: the conversion instruction; the
          // offset integer may need 33 bits (sums up to 2^31)
          load();
#pragma unroll
          for (int j = 0; j < kLd; ++j) {
            const long long v = (long long)__float2int_rn(__uint_as_float(a[j]) * scale) + kMagicI;
            acc[kLd * cb + j] += (long long)((unsigned long long)v << mult_log);
          }
        } else if (high) {
#pragma unroll
          for (int j = 0; j < kLd; ++j)
            acc[kLd * cb + j] += (long long)((unsigned long long)(a[j] * (uint32_t)mult) << 32);
        } else {
#pragma unroll
          for (int j = 0; j < kLd; ++j) acc[kLd * cb + j] += (long long)(int)a[j] * mult;
        }
      }
      bias += (long long)((unsigned long long)kMagicI << mult_log);
      tc_fence_before();
      __syncwarp();
      // the slot may be overwritten from here on
      if (lane == 0) mbar_arrive(acce + 8 * q);
      return true;
    };
    // the slot reads of one piece of a group, in the order the issuer commits
    auto drain_piece = [&](auto grp, int k0, int k1) -> bool {
      using Sc = decltype(grp);
      OzHandover<Sc> H(k0, ord);
      for (int last = 0; last < Sc::NE;) {
        int t;
        int e = H.next(t);
        const bool mid = t < k1;
        if (!mid) e = last++;
        if (!drain_slot(H.slot(e), Sc::scale_log(e), Sc::mult_log(e, p.shift_top))) return false;
        if (mid) H.move(e);
      }
      ord = H.end();
      return true;
    };
    for (int item = blockIdx.x; item < p.ntiles && ok; item += gridDim.x) {
      int tm, tn, n0;
      item_tile<NT>(p, item, tm, tn, n0);
      if (NT < OBN && n0 >= p.N) continue;
      const int m0 = tm * OBM;
      // beta C is read only when the tile is written out, after all of its
      // MMAs; fetch this thread's C entries into L2 now, so that those reads
      // wait on L2 rather than on DRAM
      if (p.prefetch_c && m0 + row < p.M) {
        const int64_t pi = m0 + row;
        for (int j = 0; j < kEpiCols; ++j) {
          const int64_t pj = n0 + kEpiCols * half + j;
          if (pj >= p.N || (p.lower && pi < pj)) break;
          asm volatile("prefetch.global.L2 [%0];" ::"l"(__cvta_generic_to_global(p.C + pi + pj * p.ldc)));
        }
      }
#pragma unroll
      for (int j = 0; j < kEpiCols; ++j) acc[j] = 0;
      if constexpr (OzDigitsOf<S>::kLow) {
        for (int c = 0; c < p.nsc && ok; ++c)
          ok = drain_piece(OzGroup<S, 0>{}, oz_piece(p.nk16, p.nsc, c),
                           oz_piece(p.nk16, p.nsc, c + 1));
        // from the unit of the lowest level to the final one
        const int d = OzDigitsOf<S>::kLowBits - p.shift_top;
        const long long b0 = bias;
        bias = 0;
        uint32_t lo16 = 0;
#pragma unroll
        for (int j = 0; j < kEpiCols; ++j) {
          acc[j] -= b0;
          if (FRAC) {
            const long long low = acc[j] & ((1ll << d) - 1);
            const uint32_t f16 = (uint32_t)(d <= 16 ? low << (16 - d) : low >> (d - 16));
            if (j & 1)
              res[(j >> 1) * (32 * kEpiWarps)] = lo16 | f16 << 16;
            else
              lo16 = f16;
            acc[j] >>= d;
          } else {
            acc[j] = (acc[j] + (1ll << (d - 1))) >> d;
          }
        }
      }
      for (int c = 0; c < p.nsc && ok; ++c)
        ok = drain_piece(OzGroup<S, 1>{}, oz_piece(p.nk16, p.nsc, c),
                         oz_piece(p.nk16, p.nsc, c + 1));
      if (!ok) break;
#pragma unroll
      for (int j = 0; j < kEpiCols; ++j) acc[j] -= bias;
      bias = 0;
      // output: alpha 2^(e_i + f_j - 2T - shift_top) acc + beta C, while
      // the MMAs of the next tile already run
      // (every lane takes part in the shuffles; rows past M store nothing)
      const int64_t gjl = n0 + kEpiCols * half + lane;
      const int f_lo = gjl < p.N ? p.eb[gjl] : 0;
      const int f_hi = kEpiCols > 32 && gjl + 32 < p.N ? p.eb[gjl + 32] : 0;
      const int64_t gi = m0 + row;
      const bool live_row = gi < p.M;
      const int ebase = live_row ? p.ea[gi] - 2 * OzDigitsOf<S>::kTop - p.shift_top : 0;
      const int64_t gj0 = n0 + kEpiCols * half;
      // Every result of this warp normal or zero, for any sum: each row's exponent far
      // enough inside the range with the least and the largest of the warp's
      // columns (a lane holds one row and two columns, the warp stores all of its
      // rows against all of its columns).
      const int em = ebase + p.alpha_exp;
      const int f_min = __reduce_min_sync(0xffffffffu, min(f_lo, f_hi));
      const int f_max = __reduce_max_sync(0xffffffffu, max(f_lo, f_hi));
      const bool inside = em + f_min > -980 && em + f_max < 940;
      const bool fast = p.alpha_pow2 && p.beta_mode < 2 && __all_sync(0xffffffffu, inside);
      // live columns of this row from gj0 on
      int64_t lim64 = (p.lower && gi + 1 < p.N ? gi + 1 : p.N) - gj0;
      const int lim = live_row ? (int)(lim64 < 0 ? 0 : (lim64 > kEpiCols ? kEpiCols : lim64)) : 0;
      double *crow = p.C + gi + gj0 * p.ldc;
      const bool add = fast && p.beta_mode == 1;
      double cv[8], cn[8];
      auto load_c = [&](int g) {
#pragma unroll
        for (int u = 0; u < 8; ++u)
          cn[u] = add && 8 * g + u < lim ? crow[(8 * g + u) * p.ldc] : 0.0;
      };
      load_c(0);
#pragma unroll
      for (int g = 0; g < kEpiCols / 8; ++g) {
#pragma unroll
        for (int u = 0; u < 8; ++u) cv[u] = cn[u];
        if (g + 1 < kEpiCols / 8) load_c(g + 1);  // in flight while this group is converted
        int f[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int cix = 8 * g + u;
          f[u] = __shfl_sync(0xffffffffu, cix < 32 ? f_lo : f_hi, cix & 31);
        }
        uint32_t rv[4] = {0, 0, 0, 0};
        if (FRAC) {
#pragma unroll
          for (int u = 0; u < 4; ++u) rv[u] = res[(4 * g + u) * (32 * kEpiWarps)];
        }
        const long long *av = acc + 8 * g;
        if (fast) {
          uint32_t fp[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) fp[u] = __byte_perm(f[2 * u], f[2 * u + 1], 0x5410);
          if (add)
            store_fast8<FRAC, true>(crow + 8 * g * p.ldc, p.ldc, lim - 8 * g, em,
                                    (uint32_t)p.alpha_neg << 31, av[0], av[1], av[2], av[3], av[4],
                                    av[5], av[6], av[7], rv[0], rv[1], rv[2], rv[3], fp[0], fp[1],
                                    fp[2], fp[3], cv[0], cv[1], cv[2], cv[3], cv[4], cv[5], cv[6],
                                    cv[7]);
          else
            store_fast8<FRAC, false>(crow + 8 * g * p.ldc, p.ldc, lim - 8 * g, em,
                                     (uint32_t)p.alpha_neg << 31, av[0], av[1], av[2], av[3], av[4],
                                     av[5], av[6], av[7], rv[0], rv[1], rv[2], rv[3], fp[0], fp[1],
                                     fp[2], fp[3], 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0);
        } else if (live_row) {
          store_out8<FRAC>(p, gi, gj0 + 8 * g, ebase, av[0], av[1], av[2], av[3], av[4], av[5], av[6],
                           av[7], rv[0], rv[1], rv[2], rv[3], f[0], f[1], f[2], f[3], f[4], f[5],
                           f[6], f[7]);
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tbase, 512);
}

// ------------------------------------------------------------- digits ----
// Row maxima of |x| as float64 bit patterns with the sign cleared (for
// non-negative float64 values the integer order is the numeric order).
// Bound by the latency of the loads: eight are in flight a thread (one at a
// time, a 6400 x 512 panel took 17 us).
__device__ __forceinline__ unsigned long long abs_bits(double x) {
  return (unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFull;
}
// exponent e of a finite m > 0 in the frexp convention, m in [2^(e-1), 2^e)
__device__ __forceinline__ int frexp_exponent(unsigned long long m) {
  const int E = (int)(m >> 52);
  return E ? E - 1022 : (64 - __clzll((long long)m)) - 1074;
}

// Scaled operands (kScaled): column k of the operand is taken times 2^t_k, t_k =
// sgn shift[k] from the other operand of the product or its own (oz_slice_rhs,
// oz_slice_inverse).  Row maxima are then kept as exponents, kKeyBias + e + t,
// which no scaling takes out of range.  A column with shift kNoTerm has no
// finite entry but 0 in the operand that set the shifts, so its terms are 0.
constexpr int kNoTerm = 1 << 24, kKeyBias = 16384;
struct Scaling {
  const int *shift;
  int sgn;
};
template <bool kScaled>
__device__ __forceinline__ unsigned long long row_key(double x, int shift, int sgn) {
  const unsigned long long m = abs_bits(x);
  if (!kScaled) return m;
  if ((m >> 52) == 0x7FF) return ~0ull;
  if (m == 0 || shift == kNoTerm) return 0;
  return (unsigned long long)(kKeyBias + frexp_exponent(m) + sgn * shift);
}
// the greatest key of x[u step], u < 8, columns k + u kstep
template <bool kScaled>
__device__ __forceinline__ unsigned long long row_key8(const double *x, int64_t step, Scaling sc,
                                                       int64_t k, int kstep,
                                                       unsigned long long mb) {
  double v[8];
  int t[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    v[u] = x[u * step];
    t[u] = kScaled ? sc.shift[k + u * kstep] : 0;
  }
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const unsigned long long b = row_key<kScaled>(v[u], t[u], sc.sgn);
    mb = b > mb ? b : mb;
  }
  return mb;
}
template <bool kScaled>
__device__ __forceinline__ unsigned long long row_key1(double x, Scaling sc, int64_t k,
                                                       unsigned long long mb) {
  const unsigned long long b = row_key<kScaled>(x, kScaled ? sc.shift[k] : 0, sc.sgn);
  return b > mb ? b : mb;
}
__device__ __forceinline__ unsigned long long warp_max(unsigned long long mb) {
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long t = __shfl_xor_sync(0xffffffffu, mb, o);
    mb = t > mb ? t : mb;
  }
  return mb;
}
// Rows strided, k contiguous: one warp per row, lanes stride over k.
template <bool kScaled>
__global__ void rowmax_kcontig_kernel(const double *X, int64_t R, int64_t K, int64_t sr,
                                      unsigned long long *bits, int Rpad, Scaling sc) {
  const int64_t r = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (r >= Rpad) return;
  unsigned long long mb = 0;
  if (r < R) {
    const double *x = X + r * sr;
    int64_t k = lane;
    for (; k + 7 * 32 < K; k += 8 * 32) mb = row_key8<kScaled>(x + k, 32, sc, k, 32, mb);
    for (; k < K; k += 32) mb = row_key1<kScaled>(x[k], sc, k, mb);
  }
  mb = warp_max(mb);
  if (lane == 0) bits[r] = mb;
}

// Rows contiguous (column-major operand): block (x, y) covers 32 rows and 256
// values of k; a warp reads 32 consecutive rows at one k (coalesced), the 8
// warps take every 8th k, and the block's maximum per row joins the others
// with atomicMax (bits zeroed beforehand).
template <bool kScaled>
__global__ void rowmax_rcontig_kernel(const double *X, int64_t R, int64_t K, int64_t sk,
                                      unsigned long long *bits, Scaling sc) {
  __shared__ unsigned long long part[8][32];
  const int rl = threadIdx.x & 31, kg = threadIdx.x >> 5;
  const int64_t r = (int64_t)blockIdx.x * 32 + rl;
  const int64_t kc0 = (int64_t)blockIdx.y * 256, kc1 = (kc0 + 256 < K) ? kc0 + 256 : K;
  unsigned long long mb = 0;
  if (r < R) {
    int64_t k = kc0 + kg;
    for (; k + 7 * 8 < kc1; k += 8 * 8)
      mb = row_key8<kScaled>(X + r + k * sk, 8 * sk, sc, k, 8, mb);
    for (; k < kc1; k += 8) mb = row_key1<kScaled>(X[r + k * sk], sc, k, mb);
  }
  part[kg][rl] = mb;
  __syncthreads();
  if (kg == 0 && r < R) {
    for (int q = 1; q < 8; ++q) mb = part[q][rl] > mb ? part[q][rl] : mb;
    if (mb) atomicMax(&bits[r], mb);
  }
}

// Shifts of an operand's columns: with m_k the largest finite |x_rk|, in [2^(e_k -
// 1), 2^e_k), and e the largest e_k, shift[k] = max(0, e - e_k - 1), kNoTerm where
// m_k = 0.  The operand's column k times 2^shift[k] against the other one's
// times 2^-shift[k] is the same product term by term; with all columns of about
// one size (within a factor of two) nothing is shifted.  The maxima and the count
// of finished blocks are zero beforehand, and the last block to finish, which
// forms the shifts, zeroes them again.  Columns run over contiguous r
// (kRowsContig): a warp a column and kColRows rows of it; else over contiguous k: a
// block 32 columns and kColRowsK rows.  Bound by latency: 16 (8) loads a thread.
constexpr int kColRows = 512, kColRowsK = 64;
template <bool kRowsContig>
__global__ void __launch_bounds__(256) column_shift_kernel(const double *X, int64_t R, int64_t K,
                                                           int64_t stride, OzColumns c) {
  __shared__ unsigned long long part[8][32];
  __shared__ int top[8];
  __shared__ bool last;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  auto finite_max = [](double x, unsigned long long mb) {
    const unsigned long long b = abs_bits(x);
    return b > mb && (b >> 52) != 0x7FF ? b : mb;
  };
  unsigned long long mb = 0;
  const int64_t step = kRowsContig ? 32 : 8 * stride;
  const int64_t k = kRowsContig ? (int64_t)blockIdx.x * 8 + warp : (int64_t)blockIdx.x * 32 + lane;
  const int64_t chunk = kRowsContig ? kColRows : kColRowsK, ro = kRowsContig ? lane : warp;
  const int rstep = kRowsContig ? 32 : 8;
  const int64_t r0 = (int64_t)blockIdx.y * chunk, r1 = r0 + chunk < R ? r0 + chunk : R;
  if (k < K) {
    const double *x = kRowsContig ? X + k * stride : X + k;
    int64_t r = r0 + ro;
    const double *p = kRowsContig ? x + r : x + r * stride;
    for (; r + 7 * rstep < r1; r += 8 * rstep, p += 8 * step) {
      double v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = p[u * step];
#pragma unroll
      for (int u = 0; u < 8; ++u) mb = finite_max(v[u], mb);
    }
    for (; r < r1; r += rstep, p += step) mb = finite_max(*p, mb);
  }
  if (kRowsContig) {
    mb = warp_max(mb);
    if (lane == 0 && mb) atomicMax(&c.kmax[k], mb);
  } else {
    part[warp][lane] = mb;
    __syncthreads();
    if (warp == 0) {
      for (int q = 1; q < 8; ++q) mb = part[q][lane] > mb ? part[q][lane] : mb;
      if (mb) atomicMax(&c.kmax[k], mb);
    }
  }
  __threadfence();
  __syncthreads();
  if (tid == 0) last = atomicAdd(c.done, 1u) + 1 == gridDim.x * gridDim.y;
  __syncthreads();
  if (!last) return;
  __threadfence();
  volatile unsigned long long *km = c.kmax;
  int e = -kNoTerm;
  for (int64_t q = tid; q < K; q += 256) {
    const unsigned long long m = km[q];
    if (m) e = max(e, frexp_exponent(m));
  }
  e = __reduce_max_sync(0xffffffffu, e);
  if (lane == 0) top[warp] = e;
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 8; ++q) e = max(e, top[q]);
  for (int64_t q = tid; q < K; q += 256) {
    const unsigned long long m = km[q];
    c.shift[q] = m ? max(0, e - frexp_exponent(m) - 1) : kNoTerm;
    km[q] = 0;
  }
  if (tid == 0) *c.done = 0;
}

// exponent e of a row from its maximum (frexp convention: every |x| < 2^e, 0 for
// a row of zeros, kNanExp for one with an infinity or a NaN)
template <bool kScaled>
__device__ __forceinline__ int exponent_of(unsigned long long m) {
  if (m == 0) return 0;
  if (kScaled) return m == ~0ull ? kNanExp : (int)m - kKeyBias;
  return (m >> 52) == 0x7FF ? kNanExp : frexp_exponent(m);
}

// x 2^sh rounded to an integer (halves away from zero) by integer operations
// on the float64 bit pattern; the caller guarantees |x| 2^sh <= 2^55
__device__ __forceinline__ long long scaled_round(double x, int sh) {
  const long long bits = __double_as_longlong(x);
  const int bexp = (int)((bits >> 52) & 0x7FF);
  unsigned long long m = (unsigned long long)(bits & ((1ll << 52) - 1));
  if (bexp != 0) m |= 1ull << 52;
  // x = m 2^(e2), e2 = max(bexp, 1) - 1075
  const int t = (bexp != 0 ? bexp : 1) - 1075 + sh;
  unsigned long long q;
  if (t >= 0)
    q = m << (t & 63);  // (t above 55 for a zero only)
  else
    q = t < -54 ? 0 : (m + (1ull << (-t - 1))) >> -t;
  return bits < 0 ? -(long long)q : (long long)q;
}

// Digits of one logical matrix X (R x K, element (r, k) at X[r sr + k sk], one
// of the strides 1) from its row maxima: block (ks, rt) writes the S tiles of
// row tile rt and K step ks, thread t the eight elements 8 (t & 1) .. of row
// t >> 1.  A warp's stores are 512 contiguous bytes per digit, and its reads
// runs of 128 bytes along whichever of r and k is contiguous.
//
// F = round(x 2^(bits - e)) + sum_i 2^7 2^(8 i) over the S - 1 low digits:
// byte i of F, less 128, is the signed digit S - i, and what is above the
// bytes is digit 1.  A byte becomes a float through the bit pattern of
// 2^23 + byte.  Digit s carries the weight 2^(-8 (s - 1)), for the two
// levels that share an accumulator.
template <int S, bool kScaled>
__global__ void __launch_bounds__(256) slice_kernel(const double *X, int64_t R, int64_t K,
                                                    int64_t sr, int64_t sk,
                                                    const unsigned long long *mx, int *e,
                                                    unsigned char *D, Scaling sc) {
  using Dg = OzDigitsOf<S>;
  const int rl = threadIdx.x >> 1, ch = threadIdx.x & 1;
  const int64_t r = (int64_t)blockIdx.y * OBM + rl, k0 = (int64_t)blockIdx.x * KS + 8 * ch;
  const int er = r < R ? exponent_of<kScaled>(mx[r]) : 0;
  if (blockIdx.x == 0 && ch == 0) e[r] = er;
  double x[8];
#pragma unroll
  for (int j = 0; j < 8; ++j)
    x[j] = (r < R && k0 + j < K && er != kNanExp) ? X[r * sr + (k0 + j) * sk] : 0.0;
  unsigned long long F[8];
  constexpr unsigned long long kBias = 0x8080808080808080ull >> (64 - 8 * (S - 1));
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    int t = 0;
    if (kScaled && k0 + j < K) {
      t = sc.shift[k0 + j];
      if (t == kNoTerm) x[j] = 0.0;
      t *= sc.sgn;
    }
    F[j] = (unsigned long long)scaled_round(x[j], Dg::kBits - er + t) + kBias;
  }
  unsigned char *dst = D + ((size_t)blockIdx.y * gridDim.x + blockIdx.x) * S * kDigitTile + rl * 32 +
                       ((ch ^ ((rl >> 2) & 1)) << 4);
#pragma unroll
  for (int s = 0; s < S; ++s) {
    // (floats with exponents down to 2^-48: exact, and exact in bf16)
    const float w = Dg::kLow ? __int_as_float((127 - 8 * s) << 23) : 1.0f;
    uint32_t o[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float f[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const unsigned long long v = F[2 * j + h];
        if (s == 0) {
          f[h] = (float)(int)((long long)v >> (8 * (S - 1)));
        } else {
          const int sh = 8 * (S - 1 - s);
          const uint32_t byte = (uint32_t)(v >> (sh & 32)) >> (sh & 31) & 0xFFu;
          f[h] = __uint_as_float(0x4B000000u | byte) - 8388736.0f;  // 2^23 + 128
        }
        if (Dg::kLow) f[h] *= w;
      }
      const __nv_bfloat162 b2 = __floats2bfloat162_rn(f[0], f[1]);
      o[j] = *(const uint32_t *)&b2;
    }
    *(uint4 *)(dst + (size_t)s * kDigitTile) = make_uint4(o[0], o[1], o[2], o[3]);
  }
}

int64_t rup(int64_t x, int64_t m) { return (x + m - 1) / m * m; }

}  // namespace

// ------------------------------------------------ shared tensor-map builder --
namespace {
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                  const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                  const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn get_encode() {
  static EncodeTiledFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (EncodeTiledFn)p;
  });
  return fn;
}
}  // namespace

bool make_map_bf16(CUtensorMap *map, const void *base, int64_t inner, int64_t rows,
                   int64_t row_bytes, int box_inner, int box_rows, int swizzle_bytes) {
  EncodeTiledFn enc = get_encode();
  if (!enc) return false;
  CUtensorMapSwizzle sw = CU_TENSOR_MAP_SWIZZLE_128B;
  if (swizzle_bytes == 64) sw = CU_TENSOR_MAP_SWIZZLE_64B;
  else if (swizzle_bytes == 32) sw = CU_TENSOR_MAP_SWIZZLE_32B;
  else if (swizzle_bytes != 128) return false;
  cuuint64_t dims[2] = {(cuuint64_t)inner, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)row_bytes};
  cuuint32_t box[2] = {(cuuint32_t)box_inner, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides,
             box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, sw,
             CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int oz_split_digits(int nslices) { return nslices <= 0 ? 6 : (nslices <= 4 ? 3 : (nslices <= 8 ? 6 : 7)); }

size_t oz_digits_bytes(int64_t R, int64_t K, int S) {
  const int64_t Rpad = rup(R, OBM), Kpad = rup(K, OBK);
  return rup((size_t)S * Rpad * Kpad * 2, 1024) + rup(12 * (size_t)Rpad, 1024);
}

OzDigits oz_digits_at(void *mem, int64_t R, int64_t K, int S) {
  const int64_t Rpad = rup(R, OBM), Kpad = rup(K, OBK);
  OzDigits d;
  d.dig = (unsigned char *)mem;
  unsigned char *x = d.dig + rup((size_t)S * Rpad * Kpad * 2, 1024);
  d.mx = (unsigned long long *)x;
  d.e = (int *)(x + 8 * (size_t)Rpad);
  d.R = R;
  d.K = K;
  d.S = S;
  return d;
}

namespace {
template <bool kScaled>
void slice_rows(const double *X, int64_t sr, int64_t sk, const OzDigits &d, Scaling sc,
                cudaStream_t st) {
  const int64_t Rpad = rup(d.R, OBM), Kpad = rup(d.K, OBK);
  if (sr == 1) {
    cudaMemsetAsync(d.mx, 0, (size_t)Rpad * sizeof(unsigned long long), st);
    dim3 g((unsigned)((Rpad + 31) / 32), (unsigned)((d.K + 255) / 256));
    rowmax_rcontig_kernel<kScaled><<<g, 256, 0, st>>>(X, d.R, d.K, sk, d.mx, sc);
  } else {
    rowmax_kcontig_kernel<kScaled>
        <<<(unsigned)((Rpad + 7) / 8), 256, 0, st>>>(X, d.R, d.K, sr, d.mx, (int)Rpad, sc);
  }
  count_launch();
  dim3 g((unsigned)(Kpad / KS), (unsigned)(Rpad / OBM));
  auto go = [&](auto kernel) {
    kernel<<<g, 256, 0, st>>>(X, d.R, d.K, sr, sk, d.mx, d.e, d.dig, sc);
  };
  if constexpr (kScaled)
    go(slice_kernel<kOzF64Digits, true>);
  else if (d.S == 3)
    go(slice_kernel<3, false>);
  else if (d.S == 6)
    go(slice_kernel<6, false>);
  else
    go(slice_kernel<7, false>);
  count_launch();
}
}  // namespace

void oz_slice(const double *X, int64_t sr, int64_t sk, const OzDigits &d, cudaStream_t st) {
  slice_rows<false>(X, sr, sk, d, Scaling{nullptr, 0}, st);
}

void oz_slice_rhs(const double *X, int64_t sr, int64_t sk, const OzDigits &d, const OzColumns &c,
                  cudaStream_t st) {
  if (sr == 1) {
    dim3 g((unsigned)((d.K + 7) / 8), (unsigned)((d.R + kColRows - 1) / kColRows));
    column_shift_kernel<true><<<g, 256, 0, st>>>(X, d.R, d.K, sk, c);
  } else {
    dim3 g((unsigned)((d.K + 31) / 32), (unsigned)((d.R + kColRowsK - 1) / kColRowsK));
    column_shift_kernel<false><<<g, 256, 0, st>>>(X, d.R, d.K, sr, c);
  }
  count_launch();
  slice_rows<true>(X, sr, sk, d, Scaling{c.shift, 1}, st);
}

void oz_slice_inverse(const double *X, int64_t sr, int64_t sk, const OzDigits &d,
                      const OzColumns &c, cudaStream_t st) {
  slice_rows<true>(X, sr, sk, d, Scaling{c.shift, -1}, st);
}

namespace {

constexpr size_t kSmemCap = 232448;  // 227 KB
constexpr int kMaxStages = 4;
template <int S>
constexpr size_t oz_smem(int nstages) {
  return 1024 + (size_t)nstages * 2 * OzDigitsOf<S>::kStageTiles * kDigitTile + kResidBytes<S> +
         (2 * nstages + 9) * 8 + 16;
}
// the deepest ring that fits (S = 6: four stages of 48 KB, S = 7: three of 56)
template <int S>
constexpr int oz_max_stages() {
  int n = kMaxStages;
  while (oz_smem<S>(n) > kSmemCap) --n;
  return n;
}
static_assert(oz_max_stages<7>() >= 3 && oz_max_stages<6>() >= 4, "ring too shallow");

// Launch attributes of an instantiation, set once: the shared-memory
// size, and the check that the warpgroups' register split (setmaxnreg) adds
// up to exactly kLaunchRegs a thread (a build that launches with any other
// count is refused rather than run: an increase that cannot be met never
// returns).  nsm: SMs of the device.
template <int S, int NT>
cudaError_t oz_prepare(int &nsm) {
  cudaError_t e = cudaFuncSetAttribute(ozaki_gemm_kernel<S, NT>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)oz_smem<S>(oz_max_stages<S>()));
  if (e != cudaSuccess) return e;
  cudaFuncAttributes fa;
  e = cudaFuncGetAttributes(&fa, ozaki_gemm_kernel<S, NT>);
  if (e != cudaSuccess) return e;
  if (NT == OBN && fa.numRegs != kLaunchRegs) return cudaErrorInvalidConfiguration;
  int dev = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  return cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
}

template <int S, int NT>
cudaError_t launch_oz_t(int reserve_sms, OzParams &p, cudaStream_t st) {
  static int nsm = 0;
  static cudaError_t prep = cudaErrorNotReady;
  static std::once_flag once;
  std::call_once(once, [] { prep = oz_prepare<S, NT>(nsm); });
  if (prep != cudaSuccess) return prep;
  // persistent: one CTA per SM (one fits: 512 TMEM columns, ~200 KB of
  // shared memory), the CTAs taking every grid-th work item; reserve_sms SMs
  // stay free for other streams
  const int cap = nsm > reserve_sms ? nsm - reserve_sms : 1;
  p.nstages = p.nstages < oz_max_stages<S>() ? p.nstages : oz_max_stages<S>();
  ozaki_gemm_kernel<S, NT>
      <<<(unsigned)(p.ntiles < cap ? p.ntiles : cap), kThreads, oz_smem<S>(p.nstages), st>>>(p);
  count_launch();
  return cudaGetLastError();
}

template <int S>
cudaError_t launch_oz(bool narrow, int reserve_sms, OzParams &p, cudaStream_t st) {
  const int rsv = reserve_sms > 0 ? reserve_sms : 0;
  return narrow ? launch_oz_t<S, kNarrow>(rsv, p, st) : launch_oz_t<S, OBN>(rsv, p, st);
}

}  // namespace

cudaError_t oz_mm(int64_t M, int64_t N, double alpha, const OzDigits &A, int64_t ra,
                  const OzDigits &B, int64_t rb, double beta_c, double *C, int64_t ldc, int lower,
                  DevStatus *status, cudaStream_t st, int reserve_sms) {
  if (M <= 0 || N <= 0) return cudaSuccess;
  const int S = A.S;
  if (B.S != S || A.K != B.K || ra % OBM || rb % OBN || ra + M > A.R || rb + N > B.R)
    return cudaErrorInvalidValue;
  const int64_t Kpad = rup(A.K, OBK);
  OzParams p;
  p.M = M;
  p.N = N;
  p.nk16 = (int)(Kpad / KS);
  const size_t rt_bytes = (size_t)p.nk16 * S * kDigitTile;
  p.DA = A.dig + (size_t)(ra / OBM) * rt_bytes;
  p.DB = B.dig + (size_t)(rb / OBN) * rt_bytes;
  p.ea = A.e + ra;
  p.eb = B.e + rb;
  const int tiles_m = (int)((M + OBM - 1) / OBM);
  p.tiles_n = (int)((N + OBN - 1) / OBN);
  {
    const int64_t ns = tune_get("ozaki_stages", kMaxStages);
    p.nstages = ns < 2 ? 2 : (ns > kMaxStages ? kMaxStages : (int)ns);
  }
  p.nsc = oz_pieces(S, p.nk16);
  p.shift_top = oz_shift_top(S, Kpad);
  p.lower = lower;
  p.alpha = alpha;
  p.betac = beta_c;
  p.beta_mode = beta_c == 0.0 ? 0 : (beta_c == 1.0 ? 1 : 2);
  p.prefetch_c = (p.beta_mode != 0 && tune_get("ozaki_prefetch_c", 1) != 0) ? 1 : 0;
  {
    int ax = 0;
    const double fr = frexp(alpha, &ax);  // alpha = fr 2^ax, |fr| in [0.5, 1)
    p.alpha_pow2 = (fr == 0.5 || fr == -0.5) ? 1 : 0;
    p.alpha_exp = ax - 1;
    p.alpha_neg = alpha < 0.0 ? 1 : 0;
  }
  p.C = C;
  p.ldc = ldc;
  p.status = status;
  p.no_loads = tune_get("test_wait_timeout", 0) != 0 ? 1 : 0;
  p.wait_ns = p.no_loads ? 1000000ull : kWaitNs;  // 1 ms in the failure-path test
  // Half-width tiles while they still fit one wave (152 SMs): the wide ones
  // would leave more than half of the SMs idle.  T Nside 16 harmonic solve 14.9
  // -> 12.8 ms, TQU Nside 8 solve 4.79 -> 4.56, 1000-map estimate 2.88 -> 2.76;
  // the same bits.
  const int tiles = oz_item_count(tiles_m, p.tiles_n, lower ? 1 : 0, 0);
  const bool narrow = 2 * tiles <= 152 - reserve_sms;
  p.ntiles = narrow ? 2 * tiles : tiles;
  p.tiles_m = tiles_m;
  {
    // bands of eight tile rows: QU Nside 32 solve 307.6 ms row by row, 292.8 in
    // bands of 4 or 8, 294.8 of 12, 295.7 of 16 (its products re-read digits from
    // DRAM); TQU Nside 16 solve (QML_FP64) 38.3, 37.9, 37.9, 37.9; products whose
    // digits stay in L2 do not change
    const int64_t b = tune_get("ozaki_band", 8);
    p.band = b < 1 ? 1 : (b > 4096 ? 4096 : (int)b);
  }
  if (S == 3) return launch_oz<3>(narrow, reserve_sms, p, st);
  if (S == 6) return launch_oz<6>(narrow, reserve_sms, p, st);
  return launch_oz<7>(narrow, reserve_sms, p, st);
}

}  // namespace qmlgb
