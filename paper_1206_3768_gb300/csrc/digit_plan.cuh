// Which tensor-core instructions a digit product issues, as plain constexpr arithmetic: the kernel
// unrolls its issue loops over these functions, the host sizes its buffers with them and a CPU
// test enumerates them.
//
// Slices s of A and t of B (from 0 here) meet at level l = s + t < S, whose accumulator is a block of
// w columns of tensor memory.  Consecutive levels form groups; for every slice s that reaches a
// group one instruction adds A's slice s times as many consecutive slices of B as the group has
// levels.  PTX orders two tcgen05.mma by their issue only if they have the same accumulator and
// the same shape; so a group is always added as a whole, by instructions of one accumulator
// address and one N, and groups share no columns.  Where a slice reaches only the upper levels of a
// group (s above the group's first level), the lower ones meet slices t < 0 of B: zeros that
// stand in front of slice 0 in every stage.
#pragma once

#ifdef __CUDACC__
#define DIGIT_FN __host__ __device__ constexpr
#else
#define DIGIT_FN constexpr
#endif

namespace digit {

constexpr int BLOCK_K = 64;          // k per K-block
constexpr int REGION = 256;          // accumulator columns of a region, two regions
constexpr int WIDEST = 64;           // widest column tile
constexpr int LARGEST_FIRST = 129;   // |digit 1|
constexpr int LARGEST_OTHER = 64;    // |digit 2 ..|

// Levels of a group.  A product of N columns takes max(N / 2, 32 + N / 4) clocks (the tensor pipe, or
// the operands' bytes out of shared memory), so N should be 128 or more, and every level more
// in a group costs up to one more product with zeros: 2 levels of 64 columns, 3 of 48, 4 of 32 or 16.
DIGIT_FN int group_levels(int S, int w) {
  const int g = w > 48 ? 2 : w > 32 ? 3 : 4;
  return g < S ? g : S;
}
// the widest tile that takes groups of g levels
DIGIT_FN int widest_with(int g) { return g == 2 ? WIDEST : g == 3 ? 48 : 32; }
DIGIT_FN int groups(int S, int g) { return (S + g - 1) / g; }
// first level of group i, S for i = groups(S, g); the first group takes the remainder of S / g
DIGIT_FN int group_begin(int S, int g, int i) { return i == 0 ? 0 : S - g * (groups(S, g) - i); }
// slices of zeros in front of slice 0 of B
DIGIT_FN int zero_slices(int g) { return g - 1; }
// Levels of region 0: all of them if they fit (region 1 then takes every other chunk), else the whole
// groups that fit, the rest being in region 1.
DIGIT_FN int region_levels(int S, int g, int w) {
  if (S * w <= REGION) return S;
  int u = 0;
  for (int i = 1; i <= groups(S, g); ++i)
    if (group_begin(S, g, i) * w <= REGION) u = group_begin(S, g, i);
  return u;
}
// The product of slice s with group i: into `levels` levels from the region's level `at` on, with as many
// slices of B from `first` on (below 0: zeros).  No levels: the slice does not reach the group.
struct Product {
  int region, at, levels, first;
};
DIGIT_FN Product product(int S, int g, int U, int s, int i) {
  const int l0 = group_begin(S, g, i), l1 = group_begin(S, g, i + 1), region = l0 >= U ? 1 : 0;
  return {region, l0 - region * U, s < l1 ? l1 - l0 : 0, l0 - s};
}
// Clocks of a K-block's products.
DIGIT_FN int block_clocks(int S, int w) {
  const int g = group_levels(S, w);
  int sum = 0;
  for (int i = 0; i < groups(S, g); ++i) {
    const int n = (group_begin(S, g, i + 1) - group_begin(S, g, i)) * w;
    sum += group_begin(S, g, i + 1) * (n / 2 > 32 + n / 4 ? n / 2 : 32 + n / 4);
  }
  return BLOCK_K / 16 * sum;
}
// Largest sum that one k can add to a level of S slices: level 0 is digit 1 squared, level l > 0 holds two
// products with a digit 1 and l - 1 without.
DIGIT_FN int largest_per_k(int S) {
  int most = LARGEST_FIRST * LARGEST_FIRST;
  for (int l = 1; l < S; ++l) {
    const int v = 2 * LARGEST_FIRST * LARGEST_OTHER + (l - 1) * LARGEST_OTHER * LARGEST_OTHER;
    if (v > most) most = v;
  }
  return most;
}
// K-blocks of an exact chunk: every integer below 2^24 is an FP32 number.
DIGIT_FN int chunk_blocks(int S) { return (1 << 24) / (largest_per_k(S) * BLOCK_K); }

}  // namespace digit
