// Powers of two that the fixed-point multipole-to-local translations
// (mc_m2l.cu) scale their operands by.  Needs only the qualifiers below, so it
// also compiles for host tests.
#pragma once

// The sums are exact, so the bits that matter are those of a matrix entry and
// of a multipole.  Both are kept as fractions of a power of two that follows
// their size, or the expansions of high degree would be left with the last
// bits only (entries fall like |o|^-(j+1): at p = 12 the highest degree came out
// 1800 times further from exact translations than in FP64 with one power for
// all, and the whole level 1700 times in a box of side 1, where that degree
// outweighs the others):
//   * offsets go by distance in MC_M2L_GROUPS groups; rows of degree j of group g are
//     2^kM2LRowScale[g][j] times the matrix's, so that no entry exceeds 1 and no row
//     sums to more than 126 over the offsets of the group (any p up to 15);
//   * columns of degree n are 2^-kM2LColScale[n] times the matrix's, the multipoles
//     2^kM2LColScale[n] times theirs: the size of a coefficient of degree n of
//     charges spread evenly over a cell;
//   * a group's sums are in units of the largest cell among the offsets of that
//     group from that target, and go to the result in FP64.
// With 9 groups every degree of the expansions of uniform charges is 0.1 to 1.0
// times as far from exact translations as in FP64 (p = 3..15, periodic and free;
// at high degrees both inherit the offset table's rounding), and with half of
// the charges in one cell 0.1 to 1.2 times.
#define MC_M2L_GROUPS 9
__host__ __device__ __forceinline__ int m2l_group(int orbit) {
  const int x = orbit & 3, y = (orbit >> 2) & 3, z = orbit >> 4, r2 = x * x + y * y + z * z;
  return (r2 >= 5) + (r2 >= 6) + (r2 >= 7) + (r2 >= 9) + (r2 >= 10) + (r2 >= 12) + (r2 >= 15) + (r2 >= 18);
}
static __constant__ signed char kM2LRowScale[MC_M2L_GROUPS][16] = {
    {1, 2, 3, 4, 5, 6, 7, 7, 8, 9, 9, 10, 10, 11, 11, 12},
    {1, 2, 3, 5, 6, 7, 9, 10, 10, 11, 12, 12, 13, 14, 14, 15},
    {1, 2, 4, 6, 7, 8, 10, 11, 12, 13, 13, 14, 15, 16, 17, 18},
    {1, 3, 5, 7, 8, 10, 11, 13, 14, 15, 17, 18, 19, 21, 22, 23},
    {1, 3, 4, 6, 7, 9, 11, 12, 14, 15, 17, 18, 20, 21, 22, 24},
    {1, 3, 5, 7, 9, 10, 12, 14, 16, 17, 19, 20, 22, 23, 25, 26},
    {1, 3, 6, 8, 10, 12, 13, 15, 17, 19, 21, 22, 24, 26, 27, 29},
    {2, 4, 7, 9, 11, 13, 15, 17, 19, 22, 23, 26, 28, 30, 32, 34},
    {2, 4, 6, 9, 11, 13, 15, 17, 19, 22, 24, 26, 28, 30, 32, 34},
};
constexpr signed char kM2LColScale[16] = {0, 2, 3, 4, 5, 6, 6, 7, 7, 8, 8, 9, 9, 10, 10, 11};
