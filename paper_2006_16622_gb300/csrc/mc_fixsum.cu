// Harmonic sums over the charges of cells in fixed point (mc_fix.cuh): the
// Alg. L.3 gather of every setup, the multipoles of Eq. (4).
#include <algorithm>
#include <mutex>

#include "mc_dev.cuh"
#include "mc_fix.cuh"
#include "mc_fixsum.cuh"

namespace {

constexpr int kRound = 256;  // source units (finest cells) listed at a time

struct FixArgs {
  FixTab tab;
  FixSource src;
  int L, l, nchunk, irregular, pbc;
  uint64_t rcp;  // fx_coord's reciprocal of the box side
  int ea;        // biased exponent of the box side
  int qexp;
  const double* dot;
  int sparse;
};

// index of a coefficient with m = 0 (no imaginary part)
__device__ __forceinline__ bool is_square_index(int k) {
  const int r = (int)sqrtf((float)k + 0.5f);
  return r * r == k;
}

__device__ __forceinline__ int64_t shfl_xor64(int64_t v, int m) {
  const int lo = __shfl_xor_sync(0xffffffffu, (int)(uint32_t)v, m);
  const int hi = __shfl_xor_sync(0xffffffffu, (int)(v >> 32), m);
  return (int64_t)(((uint64_t)(uint32_t)hi << 32) | (uint32_t)lo);
}

// Sums over the lanes of 2 x 16 terms, divided by 16: lane c ends with term
// c & 15 of ar (lanes 0..15) or ai (16..31); each exchange halves the terms a
// lane carries, and each but the first halves the terms themselves, which
// makes room for the sum; of two lanes that exchange, one rounds an odd term
// down and the other up.  (All five bits at once, before the first exchange,
// would round 32 terms at the last unit instead of two: the sums' largest
// error by far.  Level 2 of 1002 charges at p = 10: degree 10 off by 8.0e-15
// of its norm so, the FP64 gather 2.7e-15.)  B: first step, terms past ST are 0.
template <int ST, int B>
__device__ __forceinline__ int64_t lane_totals(const int64_t (&ar)[ST], const int64_t (&ai)[ST], int lane) {
  int64_t v[16];
#pragma unroll
  for (int i = 0; i < 16; i++) {
    if (B + i < ST) {
      const bool up = lane & 16;
      v[i] = (up ? ai[B + i] : ar[B + i]) + shfl_xor64(up ? ar[B + i] : ai[B + i], 16);
    } else {
      v[i] = 0;
    }
  }
#pragma unroll
  for (int w = 8; w >= 1; w >>= 1) {
#pragma unroll
    for (int i = 0; i < 2 * w; i++)
      if (B + i < ST) v[i] = (v[i] + (lane & w ? 1 : 0)) >> 1;
#pragma unroll
    for (int i = 0; i < w; i++) {
      if (B + i < ST) {
        const bool up = lane & w;
        const int64_t hi = B + i + w < ST ? v[i + w] : 0;
        v[i] = (up ? hi : v[i]) + shfl_xor64(up ? v[i] : hi, w);
      }
    }
  }
  return v[0];
}

constexpr int kThreads = 32 * MC_FIX_WARPS;
// registers: 4 per step for the sums, about 70 for the rest
constexpr int fix_ctas(int st) { return st <= 14 ? 4 : (st <= 23 ? 3 : 2); }

}  // namespace

// One CTA per (target cell, chunk of its source units).  Its four warps share
// the columns m evenly, and every lane takes one charge of a group of 32: a
// warp's table entries are uniform, no lane idles (groups of 8 lanes per
// charge leave 21 of 112 idle at p = 12), every sub-partition has the same
// work, and each lane keeps the sums of its coefficients in registers.  The
// CTA forms what depends on the displacement for 128 charges at a time, one
// per thread, in shared memory, where all four warps read it.
// Bound by the issue of integer instructions: 107 cycles of a sub-partition per
// coefficient and 32 charges, 78 of them for 18 multiply-adds of 64 bits.  One
// level of N = 1e5, p = 12 takes 4.7 ms; the same sums in FP64 (64 cycles an
// instruction) took 41 ms.
template <int P>
__global__ void __launch_bounds__(kThreads, fix_ctas(fix_shares(P).steps))
    k_fix_sums(const __grid_constant__ FixArgs A, double* __restrict__ out) {
  constexpr int ST = fix_shares(P).steps;
  constexpr int p = P, nthr = kThreads;
  __shared__ FixStep s_step[MC_FIX_WARPS][ST];
  __shared__ int s_cell[kRound], s_shift[kRound], s_pre[kRound + 1];
  extern __shared__ int64_t dyn[];
  if (A.src.range && !fix_usable(A.src.range)) return;
  const int nchunk = A.src.range ? A.src.range[3] : A.nchunk;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (A.sparse) {
    // a cell without charges has no multipole, and nothing to contract (cells
    // of up to 64 finest ones; 4096 charges at L = 7, p = 8, multipole method,
    // whole energy: 14.4 -> 8.6 ms)
    const int c = blockIdx.x / A.nchunk, n = 1 << (A.l - 1), b = A.L - A.l;
    bool any = b > 2;
    if (b <= 2 && tid < 1 << (3 * b)) {
      const int x = ((c / (n * n)) << b) + (tid >> (2 * b)), y = (((c / n) % n) << b) + ((tid >> b) & ((1 << b) - 1)),
                z = ((c % n) << b) + (tid & ((1 << b) - 1)), m = 1 << (A.L - 1);
      any = A.src.count[(x * m + y) * m + z] > 0;
    }
    if (!__syncthreads_or(any)) {
      if (tid == 0) out[blockIdx.x] = 0.0;
      return;
    }
  }
  for (int i = tid; i < MC_FIX_WARPS * ST; i += nthr) s_step[i / ST][i % ST] = A.tab.step[i / ST][i % ST];
  const bool irr = A.irregular != 0, pbc = A.pbc != 0;
  const int qexp = A.src.range ? A.src.range[1] - 1022 : A.qexp;
  int64_t* s_zeta = dyn;                 // [nthr]
  int64_t* s_kap = dyn + nthr;           // [nthr]
  int64_t* s_Y = dyn + 2 * (size_t)nthr;  // [3 (p + 1)][nthr]: Y_m^m, cos m phi, sin m phi
  const int l = A.l, nl = 1 << (l - 1), nL = 1 << (A.L - 1), fb = A.L - l, f = 1 << fb;
  const int task = blockIdx.x, t = task / A.nchunk, ch = task % A.nchunk;
  const int tc[3] = {t / (nl * nl), (t / nl) % nl, t % nl};
  const int par[3] = {tc[0] & 1, tc[1] & 1, tc[2] & 1};
  uint64_t T[3];
#pragma unroll
  for (int d = 0; d < 3; d++) T[d] = (uint64_t)(2 * tc[d] + 1) << (62 - l);
  const long long units = (long long)(irr ? 189 : 1) << (3 * fb);
  if (ch >= nchunk) return;
  const long long per = (units + nchunk - 1) / nchunk;
  const long long ub = (long long)ch * per, ue = ub + per < units ? ub + per : units;
  // steps where a column begins, from ballots so that the branch is uniform
  const unsigned turn_lo = __ballot_sync(0xffffffffu, (A.tab.turn[warp] >> lane) & 1ull);
  const unsigned turn_hi = __ballot_sync(0xffffffffu, (A.tab.turn[warp] >> (lane + 32)) & 1ull);
  int64_t ar[ST], ai[ST];
#pragma unroll
  for (int i = 0; i < ST; i++) ar[i] = ai[i] = 0;
  double sum[3] = {0.0, 0.0, 0.0};  // this lane's coefficients: steps (lane & 15) + 16 b
  int held = 0;                     // groups since the last flush
  auto flush = [&]() {
#pragma unroll
    for (int i = 0; i < ST; i++) {
      ar[i] = (ar[i] + (lane >> 4)) >> 1;
      ai[i] = (ai[i] + (lane >> 4)) >> 1;
    }
    sum[0] += (double)lane_totals<ST, 0>(ar, ai, lane);
    if constexpr (ST > 16) sum[1] += (double)lane_totals<ST, 16>(ar, ai, lane);
    if constexpr (ST > 32) sum[2] += (double)lane_totals<ST, 32>(ar, ai, lane);
#pragma unroll
    for (int i = 0; i < ST; i++) ar[i] = ai[i] = 0;
    held = 0;
  };
  for (long long u0 = ub; u0 < ue; u0 += kRound) {
    __syncthreads();
    for (int i = tid; i < kRound; i += nthr) {
      int cnt = 0, cell = 0, sh = 0;
      const long long u = u0 + i;
      if (u < ue) {
        int o[3] = {0, 0, 0};
        if (irr) il_entry((int)(u >> (3 * fb)), par, o);
        const int fc = (int)(u & (((long long)1 << (3 * fb)) - 1));
        const int fd[3] = {fc >> (2 * fb), (fc >> fb) & (f - 1), fc & (f - 1)};
        int g[3];
        bool ok = true;
#pragma unroll
        for (int d = 0; d < 3; d++) {
          const int e = tc[d] + o[d], s = mc_wrap_coord(e, nl);
          if (!pbc && e != s) ok = false;
          sh |= ((e - s) / nl + 2) << (4 * d);
          g[d] = s * f + fd[d];
        }
        cell = (g[0] * nL + g[1]) * nL + g[2];
        if (ok) cnt = A.src.start ? A.src.start[cell + 1] - A.src.start[cell] : A.src.count[cell];
      }
      s_cell[i] = cell;
      s_shift[i] = sh;
      s_pre[i + 1] = cnt;
    }
    __syncthreads();
    if (warp == 0) {
      constexpr int kPer = kRound / 32;
      int c[kPer], tot = 0;
#pragma unroll
      for (int i = 0; i < kPer; i++) {
        c[i] = s_pre[1 + lane * kPer + i];
        tot += c[i];
      }
      int inc = tot;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += v;
      }
      int run = inc - tot;
#pragma unroll
      for (int i = 0; i < kPer; i++) {
        run += c[i];
        s_pre[1 + lane * kPer + i] = run;
      }
      if (lane == 0) s_pre[0] = 0;
    }
    __syncthreads();
    const int total = s_pre[kRound];
    for (int b0 = 0; b0 < total; b0 += nthr) {
      const int idx = b0 + tid;
      FixCharge c = {0, 0, 0, 0, 0, 0};
      if (idx < total) {
        int lo = 0;
#pragma unroll
        for (int s = kRound / 2; s > 0; s >>= 1)
          if (s_pre[lo + s] <= idx) lo += s;
        const int cell = s_cell[lo], slot = idx - s_pre[lo], sh = s_shift[lo];
        double x[3], q;
        if (A.src.start) {
          const double* r = A.src.rows + 4 * ((size_t)A.src.start[cell] + slot);
          x[0] = r[0];
          x[1] = r[1];
          x[2] = r[2];
          q = r[3];
        } else {
          const double4 r = ldcg4(reinterpret_cast<const double4*>(A.src.rows) + (size_t)cell * A.src.cap + slot);
          x[0] = r.x;
          x[1] = r.y;
          x[2] = r.z;
          q = r.w;
        }
        int64_t D[3];
#pragma unroll
        for (int d = 0; d < 3; d++) {
          const int im = ((sh >> (4 * d)) & 15) - 2;
          const uint64_t X = (uint64_t)fx_coord(x[d], A.rcp, A.ea) + ((uint64_t)(int64_t)im << 62);
          const int64_t v = (int64_t)(X - T[d]);
          const int k = irr ? l - 3 : l - 1;
          D[d] = k >= 0 ? (int64_t)((uint64_t)v << k) : v >> 1;
        }
        const int64_t qf = fx_charge(q, 1023 + qexp);
        c = irr ? fix_irregular(D[0], D[1], D[2], qf) : fix_regular(D[0], D[1], D[2], qf);
      }
      s_zeta[tid] = c.zeta;
      s_kap[tid] = (int64_t)c.kap;
      {
        const Fx ex = fx_split(c.ex), ey = fx_split(c.ey), en = fx_split(-c.ey), st = fx_split(c.st);
        int64_t y = c.x0, xr = (int64_t)1 << 62, xi = 0;
        int64_t* o = s_Y + tid;
        for (int m = 0; m <= p; m++) {
          o[0] = y;
          o[nthr] = xr >> MC_FIX_PHASE;
          o[2 * nthr] = xi >> MC_FIX_PHASE;
          o += 3 * nthr;
          const Fx a = fx_split(xr), b = fx_split(xi);
          y = fx_mul62(fx_split(y), st);
          fx_turn(a, b, ex, ey, en, &xr, &xi);
        }
      }
      __syncthreads();
      const int ng = min(MC_FIX_WARPS, (total - b0 + 31) >> 5);
      if (held + ng > MC_FIX_FLUSH) flush();
      for (int g = 0; g < ng; g++) {
        const int s = g * 32 + lane;
        const uint64_t kap = (uint64_t)s_kap[s];
        const uint32_t kh = (uint32_t)(kap >> 32), kl = (uint32_t)kap;
        const Fx zp = fx_split(s_zeta[s]), zm = fx_split(-s_zeta[s]);
        Fx zs = zp, zn = zm;  // +zeta and -zeta, by step in turn
        Fx Xr = {0, 0}, Xi = {0, 0}, q1 = {0, 0}, q2 = {0, 0};
        int c = 0;
#pragma unroll
        for (int i = 0; i < ST; i++) {
          if ((i < 32 ? turn_lo >> i : turn_hi >> (i & 31)) & 1u) {  // a column begins
            const int64_t* o = s_Y + (size_t)(3 * A.tab.col[warp][c++]) * nthr + s;
            q1 = fx_split(o[0]);
            q2 = {0, 0};
            Xr = fx_split(o[nthr]);
            Xi = fx_split(o[2 * nthr]);
            zs = (i & 1) ? zm : zp;
            zn = (i & 1) ? zp : zm;
          } else {
            const FixStep st = s_step[warp][i];
            const Fx q = fix_next((i & 1) ? zs : zn, kh, kl, q1, q2, st.wh, st.wl, st.sh);
            q2 = q1;
            q1 = q;
          }
          ar[i] = fix_mac(Xr, q1, ar[i]);
          ai[i] = fix_mac(Xi, q1, ai[i]);
        }
      }
      held += ng;
      __syncthreads();
    }
  }
  flush();
  constexpr int C = (P + 1) * (P + 1);
  const double sc = ldexp(1.0, qexp);
  double* o = out + ((size_t)t * A.nchunk + ch) * C;
  double contracted = 0.0;
#pragma unroll
  for (int b = 0; 16 * b < ST; b++) {
    const int i = 16 * b + (lane & 15), im = lane >> 4;
    const int k = i < ST ? A.tab.index[warp][i] : -1;
    if (k < 0 || (im && is_square_index(k))) continue;
    double r = sum[b] * A.tab.scale[warp][i] * sc;
    if (im) r = -r;
    if (A.dot) {
      contracted += (is_square_index(k) ? 1.0 : 2.0) * r * A.dot[(size_t)t * C + k + im];
    } else {
      o[k + im] = r;
    }
  }
  if (A.dot) {
    __shared__ double part[MC_FIX_WARPS];
    contracted = warp_sum(contracted);
    if (lane == 0) part[warp] = contracted;
    __syncthreads();
    if (tid == 0) out[blockIdx.x] = (part[0] + part[1]) + (part[2] + part[3]);
  }
}

// chunk partials of many chunks and few targets: 8 warps take every eighth
// chunk of 32 coefficients, added in one order
__global__ void __launch_bounds__(256)
    k_fix_reduce(int nchunk, int C, const double* __restrict__ in, double* __restrict__ out) {
  __shared__ double s[8][32];
  const int nb = (C + 31) / 32, t = blockIdx.x / nb, k = (blockIdx.x % nb) * 32 + (threadIdx.x & 31);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double v = 0.0;
  if (k < C)
    for (int ch = warp; ch < nchunk; ch += 8) v += in[((size_t)t * nchunk + ch) * C + k];
  s[warp][lane] = v;
  __syncthreads();
  if (warp == 0 && k < C) {
    for (int w = 1; w < 8; w++) v += s[w][lane];
    out[(size_t)t * C + k] = v;
  }
}

// ------------------------------------------------------ near pairs (energy)
// q_i q_j / r_ij over the pairs of a cell with itself and with 13 of its 26
// neighbours (the other 13 see the pair from their side).  One warp per tile of
// 128 x 128 pairs of a (cell, neighbour): a lane per charge of the cell, the
// neighbour's charges staged in shared memory and read by all lanes (or, where
// few of the tile's charges are left, by the group of lanes whose turn they
// are: 4.00 -> 3.20 ms for 1e6 charges, 30.5 a cell, and 121 -> 70 us for 3e4,
// 7.3 a cell; 3.26 ms and 99 us since the sums keep their rounding).  The first
// tiles of all (cell, neighbour) come first; where
// cells may hold more than a tile, the others are counted by k_near_extra and
// dealt out in order, in tiles of 64 x 64 (4000 of 8000 charges in one cell, L =
// 5, whole fresh energy: 79 ms with one warp for a (cell, neighbour), 1.25 with
// tiles of 128 and a second look at whole tiles, 0.77 now, 0.78 with the FP64
// kernel's warp per charge; half of 16000: 1.9, 1.4 and 3.1 with the latter
// three).  At
// 30.5 a cell 310 cycles of a sub-partition for 32 pairs, idle lanes included;
// the FP64 multiply-add takes 64 beside the integer ones.  Differences are exact
// 64-bit integers; 1/r comes from a single-precision estimate and one
// third-order step in integers on the difference shifted up to full length,
// good to 2^-60, so only the last multiply-add is an FP64 instruction (one
// against 15 of a pair in FP64 at 64 cycles each).
struct NearArgs {
  FixSource src;
  int L, pbc;
  uint64_t rcp[2];  // fx_cells' reciprocal of the box side
  int ea;
  uint64_t box;  // the box side in units of 2^-60 finest cells, modulo 2^64
  double a;
  double unit;  // 1 / (four finest cells)
  int tile;  // MC_NEAR_TILE, or MC_NEAR_DENSE
  // tiles beyond the first ones, of every cell and of every 1024 cells (null:
  // no cell can hold more than a tile)
  const long long *cells, *blocks;
};
// Tiles where cells may hold more than MC_NEAR_TILE charges: a warp takes 42 us
// for one of 64 x 64, 170 for one of 128 x 128, which was the time of the kernel
// for a few thousand charges (smaller ones cost more to find than they save)
#define MC_NEAR_DENSE 64
constexpr int kNearBlock = 1024;  // cells counted by a block of k_near_extra

// neighbour o (0: itself, else one of 13) of a cell: its index, image shifts,
// and whether it exists
__device__ __forceinline__ bool near_neighbour(int cell, int o, int nL, bool pbc, int* other, int* im) {
  const int c[3] = {cell / (nL * nL), (cell / nL) % nL, cell % nL}, k = 13 + o;
  const int e[3] = {c[0] + k / 9 - 1, c[1] + (k / 3) % 3 - 1, c[2] + k % 3 - 1};
  int src[3];
  bool ok = true;
#pragma unroll
  for (int d = 0; d < 3; d++) {
    src[d] = mc_wrap_coord(e[d], nL);
    im[d] = (e[d] - src[d]) / nL;
    if (!pbc && im[d]) ok = false;
  }
  *other = (src[0] * nL + src[1]) * nL + src[2];
  return ok;
}
// tiles of (cell, neighbour o) beyond the first
__device__ __forceinline__ long long near_extra(const NearArgs& A, int cell, int o, int nL) {
  int other, im[3];
  if (o >= 14 || !near_neighbour(cell, o, nL, A.pbc, &other, im)) return 0;
  return max(near_tiles(A.src.count[cell], A.src.count[other], o == 0, A.tile) - 1, 0ll);
}

__global__ void __launch_bounds__(kNearBlock)
    k_near_extra(const __grid_constant__ NearArgs A, long long* __restrict__ cells, long long* __restrict__ blocks) {
  __shared__ long long part[kNearBlock / 32];
  const int nL = 1 << (A.L - 1), cell = blockIdx.x * kNearBlock + threadIdx.x;
  long long v = 0;
  if (cell < nL * nL * nL) {
    for (int o = 0; o < 14; o++) v += near_extra(A, cell, o, nL);
    cells[cell] = v;
  }
  for (int m = 16; m; m >>= 1) v += shfl_xor64(v, m);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kNearBlock / 32; w++) v += part[w];
    blocks[blockIdx.x] = v;
  }
}

// entry of 32 (one per lane) that item e of their sum lies in, the items
// before it taken off e; 32 if e lies beyond them all
__device__ __forceinline__ int near_find(long long v, long long* e) {
  const int lane = threadIdx.x & 31;
  long long inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const long long u = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += u;
  }
  const unsigned past = __ballot_sync(0xffffffffu, inc > *e);
  const int k = past ? __ffs(past) - 1 : 32;
  const long long before = __shfl_sync(0xffffffffu, inc - v, k & 31), all = __shfl_sync(0xffffffffu, inc, 31);
  *e -= k < 32 ? before : all;
  return k;
}
// cell, neighbour and tile of extra tile e (all lanes the same); false beyond
// the last one
__device__ __noinline__ bool near_locate(const NearArgs& A, long long e, int nL, int* cell, int* o, long long* tile) {
  const int lane = threadIdx.x & 31, ncell = nL * nL * nL, nb = (ncell + kNearBlock - 1) / kNearBlock;
  int b = 32;
  for (int b0 = 0; b0 < nb && b == 32; b0 += 32) {
    b = near_find(b0 + lane < nb ? A.blocks[b0 + lane] : 0ll, &e);
    if (b < 32) {
      for (int c0 = (b0 + b) * kNearBlock; c0 < (b0 + b + 1) * kNearBlock; c0 += 32) {
        const int k = near_find(c0 + lane < ncell ? A.cells[c0 + lane] : 0ll, &e);
        if (k == 32) continue;
        *cell = c0 + k;
        *o = near_find(near_extra(A, *cell, lane, nL), &e);
        *tile = 1 + e;
        return *o < 14;
      }
      return false;
    }
  }
  return false;
}

// Pairs closer than this (leading zeros of the difference with 2^62 = four
// finest cells, so 2^-9 of them in every component) take their distance from
// the coordinates themselves.  The two coordinates of a difference are rounded
// down by up to 2^-60 of a cell, which is 2^-54 (rms) of the distance at this
// line, as much as the FP64 operations of the other route; with the line at
// 2^-12 it was 2^-51, and 2^(L-3) times that with coordinates in 2^-62 of the
// box.  One own cell in a thousand at 24 charges a cell has such a pair; it is
// left to a second look at the block of 32 x 32 pairs (a call in the loop cost a fifth of the
// kernel).
constexpr int kNearClose = 9;
__device__ __forceinline__ int near_zeros(int64_t dx, int64_t dy, int64_t dz) {
  return __clzll((long long)((uint64_t)(dx < 0 ? -dx : dx) | (uint64_t)(dy < 0 ? -dy : dy) | (uint64_t)(dz < 0 ? -dz : dz))) - 2;
}

// 1/|(x, y, z)| for a non-zero difference in units of 2^-62 (times the caller's unit)
// and the difference's leading zeros
__device__ __forceinline__ double near_rinv(int64_t dx, int64_t dy, int64_t dz, int* zeros) {
  const int k = near_zeros(dx, dy, dz);
  *zeros = k;
  const Fx x = fx_split((int64_t)((uint64_t)dx << k)), y = fx_split((int64_t)((uint64_t)dy << k)),
           z = fx_split((int64_t)((uint64_t)dz << k));
  const int64_t n2 = fx_norm(x, y, z);  // 2^60, in [1/4, 3)
  const float yf = rsqrtf((float)(int32_t)(n2 >> 32) * 3.7252902984619140625e-9f);
  const int32_t yi = (int32_t)(yf * 536870912.0f);  // 2^29
  const uint64_t y2 = (uint64_t)((int64_t)yi * yi);
  const uint64_t plo = y2 * (uint64_t)n2, phi = __umul64hi(y2, (uint64_t)n2);
  const int64_t e = -(int64_t)((phi << 26) | (plo >> 38));  // 1 - y^2 n2 (2^80)
  const int32_t eh = (int32_t)(e >> 32);
  const int64_t c = (e >> 1) + ((3 * (((int64_t)eh * eh) >> 16)) >> 3);
  const uint64_t r = (uint64_t)(((int64_t)yi << 32) + (fx_mulint(yi, fx_split(c)) >> 16));  // 2^61, in (0.57, 2]
  // to a double: 53 leading bits, rounded; value r 2^(k - 61)
  const int s = __clzll((long long)r);  // 1, 2 or 3
  const uint64_t f = (r << s) + (1ull << 10);  // below 2^10: rounded up to the next power of two
  const uint64_t top = f < (1ull << 10) ? (1ull << 63) : f;
  const int ex = 1023 + 63 - s - 61 + k + (f < (1ull << 10) ? 1 : 0);
  return __longlong_as_double((long long)(((uint64_t)ex << 52) | ((top >> 11) & 0xFFFFFFFFFFFFFull)));
}

// a coordinate in units of 2^-60 finest cells, modulo 2^64, of an image
__device__ __forceinline__ int64_t near_coord(const NearArgs& A, double x, int image) {
  return (int64_t)((uint64_t)fx_cells(x, A.rcp[0], A.rcp[1], A.ea, A.L) + (uint64_t)(int64_t)image * A.box);
}
__device__ __forceinline__ int64_t near_diff(int64_t xi, int64_t xj) { return (int64_t)((uint64_t)xi - (uint64_t)xj); }

// q_i q_j / r (in the kernel's unit) over this lane's close pairs of charges
// i0..i1 of a cell and j0..j1 of another (the same one: j < i)
__device__ __noinline__ double near_close_pairs(const NearArgs& A, const double4* u, int i0, int i1, const double4* v,
                                                int j0, int j1, int im) {
  const int ix = (im & 3) - 1, iy = ((im >> 2) & 3) - 1, iz = (im >> 4) - 1;
  double acc = 0.0;
  for (int i = i0 + (threadIdx.x & 31); i < i1; i += 32) {
    const double4 x = ldcg4(&u[i]);
    const int je = u == v ? min(i, j1) : j1;
    for (int j = j0; j < je; j++) {
      const double4 y = ldcg4(&v[j]);
      // the image's coordinate is t + i a; the sum that is exact comes first
      auto diff = [&](double s, double t, int i) { return i > 0 ? (s - A.a) - t : s - (t + i * A.a); };
      auto fixed = [&](double s, double t, int i) { return near_diff(near_coord(A, s, 0), near_coord(A, t, i)); };
      if (near_zeros(fixed(x.x, y.x, ix), fixed(x.y, y.y, iy), fixed(x.z, y.z, iz)) < kNearClose) continue;
      const double dx = diff(x.x, y.x, ix), dy = diff(x.y, y.y, iy), dz = diff(x.z, y.z, iz);
      acc += x.w * y.w / (sqrt(dx * dx + dy * dy + dz * dz) * A.unit);
    }
  }
  return acc;
}

__global__ void __launch_bounds__(256, 4)
    k_fix_near(const __grid_constant__ NearArgs A, double* __restrict__ out) {
  __shared__ int64_t s_x[8][32][4];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nL = 1 << (A.L - 1), cap = A.src.cap;
  const long long tasks = 14LL * nL * nL * nL;
  const double4* rows = reinterpret_cast<const double4*>(A.src.rows);
  double total = 0.0, low = 0.0;  // the sum and its rounding
  for (long long task = (long long)blockIdx.x * 8 + warp;; task += (long long)gridDim.x * 8) {
    int cell = (int)(task / 14), o = (int)(task % 14), ti = 0, tj = 0;  // o = 0: the cell itself
    long long tile = 0;
    if (task >= tasks && !(A.cells && near_locate(A, task - tasks, nL, &cell, &o, &tile))) break;
    int other, im[3];
    if (!near_neighbour(cell, o, nL, A.pbc, &other, im)) continue;
    int ni = A.src.count[cell], nj = A.src.count[other];
    if (tile) near_tile(tile, nj, o == 0, &ti, &tj, A.tile);
    const int ib = ti * A.tile, jb = tj * A.tile;
    ni = min(ni, ib + A.tile);
    nj = min(nj, jb + A.tile);
    unsigned close = 0;  // blocks of 32 x 32 pairs with close ones (bit 4 row + column)
    for (int i0 = ib; i0 < ni; i0 += 32) {
      // fewer than 17 particles left: 2 to 32 groups of lanes share the other
      // cell's particles (at 30.5 a cell a second pass has five on average)
      const int sh = ni - i0 > 16 ? 5 : 32 - __clz(ni - i0 - 1);
      const int i = i0 + (lane & ((1 << sh) - 1));
      int64_t xi[3] = {0, 0, 0};
      double qi = 0.0, acc = 0.0;
      if (i < ni) {
        const double4 r = ldcg4(&rows[(size_t)cell * cap + i]);
        xi[0] = near_coord(A, r.x, 0);
        xi[1] = near_coord(A, r.y, 0);
        xi[2] = near_coord(A, r.z, 0);
        qi = r.w;
      }
      for (int j0 = jb; j0 < nj; j0 += 32) {
        if (o == 0 && j0 > i0) break;  // pairs i > j
        __syncwarp();
        if (j0 + lane < nj) {
          const double4 r = ldcg4(&rows[(size_t)other * cap + j0 + lane]);
          int64_t* x = s_x[warp][lane];
          x[0] = near_coord(A, r.x, im[0]);
          x[1] = near_coord(A, r.y, im[1]);
          x[2] = near_coord(A, r.z, im[2]);
          x[3] = __double_as_longlong(r.w);
        }
        __syncwarp();
        const int jn = min(32, nj - j0);
        bool here = false;
        // eight pairs at a time, so that the running sum rounds at an eighth of
        // the additions: a pair counts once here, in the FP64 kernel from both
        // sides, which averages the rounding of two sums.  Energies of 2000
        // charges at L = 3: 9.0e-14 (rms) off with one running sum and plain sums
        // after it, 4.1e-14 now, FP64 5.4e-14
        for (int j = lane >> sh; j < jn;) {
          const int je = min(jn, j + (8 << (5 - sh)));
          double part = 0.0;
#pragma unroll 1
          for (; j < je; j += 32 >> sh) {
            const int64_t* x = s_x[warp][j];
            if (i >= ni || (o == 0 && j0 + j >= i)) continue;
            int64_t d[3];
#pragma unroll
            for (int a = 0; a < 3; a++) d[a] = near_diff(xi[a], x[a]);
            int k;
            const double rinv = near_rinv(d[0], d[1], d[2], &k);
            here |= k >= kNearClose;
            // (rinv is finite for any difference)
            part = fma(k >= kNearClose ? 0.0 : __longlong_as_double(x[3]), rinv, part);
          }
          acc += part;
        }
        if (here) close |= 1u << ((i0 - ib) / 32 * 4 + (j0 - jb) / 32);
      }
      two_add(&total, &low, qi * acc);
    }
    for (close = __reduce_or_sync(0xffffffffu, close); close; close &= close - 1) {
      const int b = __ffs(close) - 1, i0 = ib + 32 * (b / 4), j0 = jb + 32 * (b % 4);
      two_add(&total, &low, near_close_pairs(A, &rows[(size_t)cell * cap], i0, min(ni, i0 + 32), &rows[(size_t)other * cap],
                                             j0, min(nj, j0 + 32), (im[0] + 1) | (im[1] + 1) << 2 | (im[2] + 1) << 4));
    }
  }
  warp_two_sum(&total, &low);
  __shared__ double s_sum[8][2];
  if (lane == 0) {
    s_sum[warp][0] = total;
    s_sum[warp][1] = low;
  }
  __syncthreads();
  if (warp > 0) return;
  total = lane < 8 ? s_sum[lane][0] : 0.0;
  low = lane < 8 ? s_sum[lane][1] : 0.0;
  warp_two_sum(&total, &low);
  if (lane == 0) {
    // times 1 / (4 w), w = a / nL
    const double x = total * (0.25 * nL), r = x / A.a;
    out[2 * blockIdx.x] = r;
    out[2 * blockIdx.x + 1] = (fma(-r, A.a, x) + low * (0.25 * nL)) / A.a;
  }
}

static int near_size(int cap) { return cap <= MC_NEAR_TILE ? MC_NEAR_TILE : MC_NEAR_DENSE; }

int fix_near_blocks(int L, int sms, int cap) {
  // a warp per tile, if every cell were full
  const double tiles = (double)(14LL << (3 * (L - 1))) * (double)near_tiles(cap, cap, false, near_size(cap));
  return (int)std::min(tiles / 8.0 + 1.0, 8.0 * sms);
}

static void box_scale(double a, uint64_t* rcp, int* ea) {
  uint64_t u;
  __builtin_memcpy(&u, &a, 8);
  *ea = (int)((u >> 52) & 0x7ff);
  const uint64_t m = (u & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull;
  *rcp = (uint64_t)((((unsigned __int128)1 << 115) + m / 2) / m);
}

size_t fix_near_work(int L, int cap) {
  const size_t ncell = (size_t)1 << (3 * (L - 1));
  return cap <= MC_NEAR_TILE ? 0 : ncell + (ncell + kNearBlock - 1) / kNearBlock;
}

cudaError_t fix_near(int L, bool pbc, double a, const FixSource& src, int blocks, double* out, cudaStream_t st) {
  NearArgs A;
  A.src = src;
  A.L = L;
  A.pbc = pbc;
  A.a = a;
  {
    uint64_t u;
    __builtin_memcpy(&u, &a, 8);
    A.ea = (int)((u >> 52) & 0x7ff);
    const uint64_t m = (u & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull;
    const unsigned __int128 top = (unsigned __int128)1 << 115;
    A.rcp[0] = (uint64_t)(top / m);
    A.rcp[1] = (uint64_t)((top % m << 64) / m);
  }
  A.box = L < 5 ? 1ull << (59 + L) : 0ull;
  A.unit = (double)(1 << (L - 1)) / (4.0 * a);
  A.tile = near_size(src.cap);
  A.cells = A.blocks = nullptr;
  if (fix_near_work(L, src.cap)) {
    const int ncell = 1 << (3 * (L - 1)), nb = (ncell + kNearBlock - 1) / kNearBlock;
    long long* cells = reinterpret_cast<long long*>(out + 2 * (size_t)blocks);
    k_near_extra<<<nb, kNearBlock, 0, st>>>(A, cells, cells + ncell);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    A.cells = cells;
    A.blocks = cells + ncell;
  }
  k_fix_near<<<blocks, 256, 0, st>>>(A, out);
  return cudaGetLastError();
}

__global__ void k_reduce_chunks(int, int, int, const double*, double*);

cudaError_t fix_reduce(int ntarget, int nchunk, int C, int sms, const double* in, double* out, cudaStream_t st) {
  // one thread per coefficient up to 8 chunks, eight warps per coefficient
  // block above
  if (nchunk <= 8) {
    const size_t b = ((size_t)ntarget * C + 255) / 256;
    k_reduce_chunks<<<(int)std::max<size_t>(1, std::min<size_t>(b, (size_t)sms * 8)), 256, 0, st>>>(ntarget, nchunk, C,
                                                                                                  in, out);
  } else {
    k_fix_reduce<<<ntarget * ((C + 31) / 32), 256, 0, st>>>(nchunk, C, in, out);
  }
  return cudaGetLastError();
}

int fix_chunks(int L, int l, bool irregular, int sms, double occupancy, int p) {
  const long long nl = 1LL << (l - 1), ncl = nl * nl * nl;
  const long long units = (irregular ? 189LL : 1LL) << (3 * (L - l));
  // about eight tasks per resident CTA ...
  const long long want = (8LL * fix_ctas(fix_shares(p).steps) * sms + ncl - 1) / ncl;
  // ... that are worth it
  static_assert(kThreads == 128, "fix_chunks_worth");
  return (int)std::max<long long>(1, std::min(want, fix_chunks_worth(units, occupancy)));
}

// Tables of an order for a radius of 1, formed on first use and never changed.
// (Where long double is software, as on Arm hosts, forming them takes 7 to 85 us,
// p = 4 to 15, which was longer than the kernels of a small system; the scales of
// a radius take a tenth of that.)
struct FixBase {
  FixTab tab;
  long double unit[MC_FIX_WARPS][MC_FIX_STEPS];
};
static const FixBase& fix_base(int p, bool irregular) {
  static FixBase base[MC_PMAX + 1][2];
  static std::once_flag once[MC_PMAX + 1][2];
  std::call_once(once[p][irregular], [&] { fix_tab_build(&base[p][irregular].tab, p, irregular, 1.0, base[p][irregular].unit); });
  return base[p][irregular];
}

cudaError_t fix_launch(const FixPass& ps, const FixSource& src, double* out, cudaStream_t st) {
  if (ps.p < 0 || ps.p > MC_PMAX) return cudaErrorInvalidValue;
  FixArgs A;
  const double w = ps.a / (double)(1 << (ps.l - 1));
  {
    const FixBase& b = fix_base(ps.p, ps.irregular);
    A.tab = b.tab;
    // R^n, or R^-(n + 1)
    const long double R = ps.irregular ? kFixR0 * w : w, step = ps.irregular ? 1.0L / R : R;
    long double power[MC_PMAX + 1];
    power[0] = ps.irregular ? step : 1.0L;
    for (int n = 1; n <= ps.p; n++) power[n] = power[n - 1] * step;
    for (int k = 0; k < MC_FIX_WARPS; k++)
      for (int t = 0; t < MC_FIX_STEPS; t++) {
        const int i = A.tab.index[k][t];
        if (i < 0) continue;
        int n = 0;
        while ((n + 1) * (n + 1) <= i) n++;
        A.tab.scale[k][t] = (double)(b.unit[k][t] * power[n]);
      }
  }
  A.src = src;
  A.L = ps.L;
  A.l = ps.l;
  A.nchunk = ps.nchunk;
  A.irregular = ps.irregular;
  A.pbc = ps.pbc;
  A.qexp = ps.qexp;
  A.dot = ps.dot;
  A.sparse = ps.dot && ps.sparse && !src.start;
  box_scale(ps.a, &A.rcp, &A.ea);
  const size_t smem = sizeof(int64_t) * (size_t)kThreads * (2 + 3 * (ps.p + 1));
  const long long ncl = 1LL << (3 * (ps.l - 1));
  const long long grid = ncl * ps.nchunk;
  if (grid > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
  cudaError_t e = cudaErrorInvalidValue;
#define MC_FIX_CASE(P_)                                                                              \
  case P_:                                                                                          \
    e = cudaFuncSetAttribute(k_fix_sums<P_>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem); \
    if (e == cudaSuccess) {                                                                         \
      k_fix_sums<P_><<<(int)grid, kThreads, smem, st>>>(A, out);                                    \
      e = cudaGetLastError();                                                                       \
    }                                                                                               \
    break;
  switch (ps.p) {
    MC_FIX_CASE(0)
    MC_FIX_CASE(1)
    MC_FIX_CASE(2)
    MC_FIX_CASE(3)
    MC_FIX_CASE(4)
    MC_FIX_CASE(5)
    MC_FIX_CASE(6)
    MC_FIX_CASE(7)
    MC_FIX_CASE(8)
    MC_FIX_CASE(9)
    MC_FIX_CASE(10)
    MC_FIX_CASE(11)
    MC_FIX_CASE(12)
    MC_FIX_CASE(13)
    MC_FIX_CASE(14)
    MC_FIX_CASE(15)
  }
#undef MC_FIX_CASE
  return e;
}
