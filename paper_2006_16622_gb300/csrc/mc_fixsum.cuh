// Launch interface of the fixed-point harmonic sums (mc_fixsum.cu).
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>

// where the charges are: rows (x, y, z, q) of finest cell c begin at
// c * cap with count[c] of them, or (start != null) at start[c] up to
// start[c + 1]
struct FixSource {
  const double* rows;
  const int* count;
  int cap;
  const int* start;
  // range of the charges found on the device (mc_noalloc.cu), or null:
  // {unusable, largest biased exponent e of a non-zero charge, largest
  // 4096 - e}, all 0 without any, and the chunks in use
  const int* range;
};

// One pass over level l (1 = the box): irregular sums over the interaction
// list of every cell, or regular sums over the cell's own charges.  Chunk ch
// of cell t goes to out[(t * nchunk + ch) * C] in the scaled layout; with
// `dot` (the level's other expansions, C per cell) only its contraction
// sum_k W_k S_k dot_k (W = 1 for m = 0, else 2) goes to out[t * nchunk + ch].
struct FixPass {
  int L, l, p;
  bool irregular, pbc;
  double a;     // box side
  int qexp;     // charges are at most 2^qexp in size
  int nchunk;   // chunks of the source units (finest cells) per target
  const double* dot;
  bool sparse;  // with dot: most finest cells are empty (of use, not of need)
};
// chunks per target that keep every SM busy without tasks too short to pay
// for themselves (occupancy: mean charges of a finest cell)
int fix_chunks(int L, int l, bool irregular, int sms, double occupancy, int p);
// the part of it that needs the occupancy: chunks of `units` finest cells with
// at least two staged batches of 128 charges each
#ifdef __CUDACC__
__host__ __device__ __forceinline__ long long fix_chunks_worth(long long units, double occupancy) {
  const double n = (double)units / (256.0 / (occupancy > 0.25 ? occupancy : 0.25));
  return n < 1.0 ? 1 : (n < (double)units ? (long long)n : units);
}
#endif
cudaError_t fix_launch(const FixPass& ps, const FixSource& src, double* out, cudaStream_t st);
// Direct part of the energy: 1/r over the pairs of charges within near cells
// (every pair and image once), one partial
// (a sum and its rounding) for each of the returned number of blocks, followed by
// the workspace of fix_near_work doubles (of use until the call's kernels are
// done)
int fix_near_blocks(int L, int sms, int cap);
size_t fix_near_work(int L, int cap);
cudaError_t fix_near(int L, bool pbc, double a, const FixSource& src, int blocks, double* out, cudaStream_t st);
// charges of this span of exponents (largest minus smallest) keep the
// fixed-point sums at least as accurate as FP64 ones
#define MC_FIX_QSPAN 6
#ifdef __CUDACC__
__host__ __device__ __forceinline__ bool fix_usable(const int* range) {
  return range[0] == 0 && range[1] + range[2] - 4096 <= MC_FIX_QSPAN;
}
#endif
// out[t][k] = sum over the chunks of target t, in one order
cudaError_t fix_reduce(int ntarget, int nchunk, int C, int sms, const double* in, double* out, cudaStream_t st);
