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

// The accumulation steps of a column block for K <= 64 and K <= 128: the
// group, and its 64-wide K chunks c0 <= c < c1. FP32 accumulation of integers
// is exact below 2^24, and the chunks keep the sums of the leading groups
// there: |a_0 b_0| <= 2^17 over 128 terms; the products of groups 1 and 2 have
// |a| <= 2^9 and, over U_k's entries, |b| of half its 2^9 on average, so their
// sums over 64 terms stay below 2^23 per product (2^22 with a_0). Group 3
// weighs 2^-30 of group 0: a rounding there is below the result's last bit.
struct Step { int g, c0, c1; };
template <int KT> struct Steps {
  static constexpr int kCount = KT > 64 ? 8 : 6;
  static constexpr Step at(int i) {
    if (KT <= 64) return Step{i, 0, 1};
    if (i == 0) return Step{0, 0, 2};
    if (i < 5) return Step{(i + 1) / 2, (i - 1) % 2, (i - 1) % 2 + 1};
    return Step{i - 2, 0, 2};
  }
};

// B's slices arrive by bulk copies on two barriers: slices below first_slices
// on barrier 0, the others on barrier 1. Bit i: the warp that issues the
// products of a step of group g has to have waited on barrier i. Steps are
// issued by different warps, and the first two with no other order between
// them, so every step waits for all that it reads.
constexpr unsigned step_waits(int KP, int g) { return 1u | (g >= first_slices(KP) ? 2u : 0u); }

}  // namespace igafd_split
