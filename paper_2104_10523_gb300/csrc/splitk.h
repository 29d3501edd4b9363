// Split-K policy shared by the planner (workspace sizing) and the executor.
//
// A step whose output has few tiles but a long contracted dimension (for
// example the final inner products of two large tensors) would otherwise run
// on a handful of CTAs.  Its K range is then split over several CTAs that
// write FP32 partial products; an ordered reduction adds them.
#pragma once

#include <algorithm>
#include <cmath>
#include <cstdint>

namespace tnq {

constexpr int kSplitTargetCtas = 2 * 152;   // aim for two waves of CTAs on the 152 SMs
constexpr double kPartialCapElems = 1 << 26;  // complex64 partial elements (512 MB)

// Skinny steps (few output rows or columns) stay on the CUDA cores even in the
// tensor-core modes: they are bandwidth-bound and a 128-row MMA tile would idle.
// Default rule (the autotuner may override it per step): steps with a small
// side of at most 16 rows are bandwidth-bound and stay on the CUDA cores.
inline bool skinny(int nM, int nN, int nK) {
  (void)nK;
  const int s = nM < nN ? nM : nN;
  return s <= 4;
}

// Flops per byte of a skinny step: 8 M K flops and 8 (M + K) bytes per row of the
// large operand.
inline double flops_per_byte(int nS, int nK) {
  const double m = std::ldexp(1.0, nS), k = std::ldexp(1.0, nK);
  return m * k / (m + k);
}

// Whether the short-K gather kernel runs the step near the memory bound: K of at
// most 32 (a row sits in registers) and a small side of at most 128 rows at no
// more than about 10 flops per byte, the FFMA rate over the memory rate (60 TF/s
// achieved, 6 TB/s).
inline bool gather_bound(int nM, int nN, int nK) {
  const int s = nM < nN ? nM : nN;
  if (nK > 5 || s > 7) return false;
  if (s <= 5) return true;  // register rows beat staged or tiled kernels even above that line
  return flops_per_byte(s, nK) <= 10.0;
}

// Tiny outputs (M, N <= 8) with a long contracted dimension never fill a
// tensor-core tile.
inline bool use_dot(int nM, int nN, int nK) { return nM <= 3 && nN <= 3 && nK >= 10; }

// tiles: CTAs without splitting; kunits: K extent in units the split may cut
// (SIMT: 16-element K slices; tensor cores: 128-byte K blocks); min_units: the
// least K units one split should keep.
inline int split_factor(double tiles, double kunits, double min_units, double out_elems) {
  int s = 1;
  while (tiles * s < kSplitTargetCtas && kunits / (2.0 * s) >= min_units && out_elems * 2.0 * s <= kPartialCapElems)
    s *= 2;
  return s;
}

inline int simt_splits(int nH, int nM, int nN, int nK) {
  double tiles = std::ldexp(1.0, nH) * std::ceil(std::ldexp(1.0, nM) / 64.0) * std::ceil(std::ldexp(1.0, nN) / 64.0);
  return split_factor(tiles, std::ceil(std::ldexp(1.0, nK) / 16.0), 16.0, std::ldexp(1.0, nH + nM + nN));
}

// Long-K kernel with a small side of at most 32 rows (kdot.cu): its tile holds
// every M index, 2^tn N values (16, 32 beside 16 or more rows) and as many K
// values as one of two 48 KB buffers takes beside them.
constexpr int kKdotTileElems = 6144;
inline bool use_kdot(int nM, int nN, int nK) { return (nM < nN ? nM : nN) <= 5 && nK >= 6; }
inline void kdot_tile(int nM, int nN, int nK, int* tn, int* tk) {
  *tn = std::min(nN, nM >= 4 ? 5 : 4);
  *tk = 6;
  while (*tk < nK && *tk < 11 && (((1 << nM) + (1 << *tn)) << (*tk + 1)) <= kKdotTileElems) ++*tk;
}
// K tiles are shared out over CTAs until two of them run on every SM.
inline int kdot_splits(int nH, int nM, int nN, int nK) {
  int tn, tk;
  kdot_tile(nM, nN, nK, &tn, &tk);
  const double units = std::ldexp(1.0, nH + nN - tn), tiles = std::ldexp(1.0, nK - tk);
  const double cap = kPartialCapElems / std::ldexp(1.0, nH + nM + nN);
  return int(std::max(1.0, std::min({std::floor(kSplitTargetCtas / units), tiles, cap})));
}

// Whether the rows kernel takes a long-K step from the long-K kernel, whose CTAs pay
// for their tables on 16 or 32 rows of the large operand: where rows (batch entries
// included) are many, K is short and a batch entry fills the rows kernel's tile of
// 128 rows (half of it at K = 64).  The table holds log2 of the rows from which, by
// log2 of the small side's rows and of K (from 6 on; 99: never); `permuted`: G is not
// stored with K lowest, so the rows kernel needs a permute first.  Time of the long-K
// kernel over the rows kernel's, call against call: K = 64, 8 x 2^20 3.0 in place
// and 2.2 permuted, 2^16 1.6 and 1.1, 2^14 0.9 and 0.6; K = 128, 8 x 2^20 1.7 and 1.2;
// K = 256, 8 x 2^19 1.1 and 0.8; K = 512, 32 x 2^18 1.1 and 0.8; below 0.8 beyond.
inline bool rows_faster(bool permuted, int nM, int nN, int nH, int nK) {
  static constexpr signed char from[2][6][5] = {{{16, 21, 99, 99, 99},
                                                 {15, 16, 99, 99, 99},
                                                 {15, 16, 19, 99, 99},
                                                 {15, 16, 19, 99, 99},
                                                 {15, 16, 99, 99, 99},
                                                 {15, 16, 17, 18, 19}},
                                                {{18, 99, 99, 99, 99},
                                                 {17, 18, 99, 99, 99},
                                                 {16, 17, 99, 99, 99},
                                                 {16, 17, 99, 99, 99},
                                                 {17, 18, 99, 99, 99},
                                                 {16, 17, 99, 99, 99}}};
  if (nM > 5 || nK < 6 || nK > 10 || nN < (nK == 6 ? 6 : 7)) return false;
  return nN + nH - (nN == 6) >= from[permuted][nM][nK - 6];
}

// Whether the rows kernel takes a long-K step whose sums keep a fixed order from the
// one-launch kernel (one lane an output, both operands uncoalesced): the same sums in
// the same order, so the choice never shows in the results.  One-lane time over
// rows time by log2 of the large operand's elements t, 2^nN rows: 16 rows of S 1.6
// at t = 21, 5.6 at 24, up to 17 at 26 (permuted first: 0.6, 1.4 to 4, 1.5 to 4.7);
// 8 rows 1.1, 3 and 8 (0.5, 0.9 to 2.2, 1 to 2.5); 4 rows 0.6, 1.6 and 4.5 (0.5, 0.6
// to 1.4, 0.7 to 1.4); 2 rows 0.6, 0.9 and 0.9, but 1.4 to 2.3 from K = 2^18 on; with
// fewer rows in S or in a batch entry of G the one-launch kernel stays ahead.
inline bool rows_ordered(bool permuted, int nM, int nN, int nH, int nK) {
  const int t = nN + nH + nK;
  if (nM >= 4) return nN >= 5 && t >= (permuted ? 23 : 21);
  if (nM == 3) return nN >= 6 && t >= (permuted ? 24 : 22);
  if (nM == 2) return !permuted && nN >= 7 && t >= 22;
  return nM == 1 && !permuted && nN >= 7 && nK >= 18;
}

// K splits of a long-K step whose sums keep a fixed order (one lane per output,
// ascending K): at least 256 K values a split.
inline int ordered_splits(int nH, int nM, int nN, int nK) {
  if (nK <= 5) return 1;
  double tiles = std::ldexp(1.0, nH) * std::ceil(std::ldexp(1.0, std::max(nM, nN)) / 128.0);
  return split_factor(tiles, std::ceil(std::ldexp(1.0, nK) / 32.0), 8.0, std::ldexp(1.0, nH + nM + nN));
}

// bf16: 64 complex elements per 128-byte K block of A'; tf32: 16.
inline int tc_splits(int nH, int nM, int nN, int nK, bool bf16) {
  double tiles = std::ldexp(1.0, nH) * std::ceil(std::ldexp(2.0, nM) / 128.0) *
                 std::ceil(std::ldexp(1.0, nN) / 256.0);
  double kblocks = std::ceil(std::ldexp(2.0, nK) / (bf16 ? 64.0 : 32.0));
  return split_factor(tiles, kblocks, 8.0, std::ldexp(1.0, nH + nM + nN));
}

}  // namespace tnq
