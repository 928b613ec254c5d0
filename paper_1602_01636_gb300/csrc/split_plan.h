// Schedule of the digit products of the split FP64 FD (fd_split.cu): plain
// constant expressions, also compiled by the host compiler in the tests.
#pragma once

namespace igafd_split {

constexpr int kSlices = 6;              // digits per operand

// With K > 128 the rows are split and multiplied in two parts (the first 128
// terms, then the rest, on the same row exponents) whose groups add up in the
// 64-bit sums.
constexpr int part_terms(int KP) { return KP > 128 ? 128 : KP; }
// slices of B fetched before the input is read (the rest of B's shared memory
// holds the transposition buffers until then)
constexpr int first_slices(int KP) { return KP > 128 ? kSlices : KP > 64 ? 3 : 1; }

// |digit| of either operand: X has 58 bits, so that its top digit is at most
// 2^8 (with the carry of the digits below), the others lie in -512 .. 511.
constexpr int kBits = 58;
constexpr long long digit_bound(int s) { return s == 0 ? 1 << (kBits - 50) : 1 << 9; }

// One accumulation step of a column block: the products a_s b_(g - s) of group
// g for the bits s of prods, over the 16-term blocks k0 <= k < k1.
struct Step {
  int g;
  unsigned prods;
  int k0, k1;
};
// largest |sum| over `terms` terms
constexpr long long step_bound(int g, unsigned prods, int terms) {
  long long b = 0;
  for (int s = 0; s <= g; ++s)
    if (prods >> s & 1u) b += digit_bound(s) * digit_bound(g - s);
  return b * terms;
}

// The steps for KT <= 128 terms. The FP32 accumulators hold integers exactly up
// to 2^24, so the sums of groups 0 to 3 are cut where the largest digits could
// pass it: 64 terms of group 1, 32 of group 2, in group 3 32 of three products
// and 64 of the fourth. Groups 4 and 5 take all terms at once: their unit is
// 2^-54 and 2^-64 of the largest a times the largest b, and cutting group 4 at
// 64 terms changed no error by a tenth of a unit of 2^-53 of the norms.
constexpr int kExact = 4;
struct StepList {
  int n = 0;
  Step s[16] = {};
};
constexpr StepList steps_of(int KT) {
  StepList l;
  for (int g = 0; g < kSlices; ++g) {
    const unsigned all = (2u << g) - 1, sets[2] = {g == 3 ? 0xbu : all, g == 3 ? 0x4u : 0u};
    for (const unsigned prods : sets) {
      if (!prods) continue;
      const int blocks = KT / 16;
      const int cut = g < kExact ? (int)((1ll << 24) / step_bound(g, prods, 16)) : blocks;
      for (int k = 0; k < blocks; k += cut) l.s[l.n++] = Step{g, prods, k, k + cut < blocks ? k + cut : blocks};
    }
  }
  return l;
}
template <int KT> struct Steps {
  static constexpr int kCount = steps_of(KT).n;
  static constexpr Step at(int i) { return steps_of(KT).s[i]; }
};
constexpr bool sums_exact(int KT) {
  const StepList l = steps_of(KT);
  for (int i = 0; i < l.n; ++i)
    if (l.s[i].g < kExact && step_bound(l.s[i].g, l.s[i].prods, 16 * (l.s[i].k1 - l.s[i].k0)) > 1ll << 24) return false;
  return l.s[0].g == 0 && (l.n < 2 || l.s[1].g != 0);    // group 0 in one step
}
static_assert(sums_exact(32) && sums_exact(64) && sums_exact(96) && sums_exact(128));

// B's slices arrive by bulk copies on two barriers: slices below first_slices
// on barrier 0, the others on barrier 1. Bit i: the warp that issues the
// products of a step of group g has to have waited on barrier i. Steps are
// issued by different warps, and the first two with no other order between
// them, so every step waits for all that it reads.
constexpr unsigned step_waits(int KP, int g) { return 1u | (g >= first_slices(KP) ? 2u : 0u); }

}  // namespace igafd_split
