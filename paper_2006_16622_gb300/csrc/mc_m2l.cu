// Multipole-to-local translations of the fast setup (Sec. 3.2, last
// paragraph) in fixed point on the integer pipe.
//
// With multipoles and expansions in units of their cell (Mhat = M w^-n,
// Lhat = L w^(j+1), paper normalisation) every offset o of an interaction
// list has one matrix T_o of size C x C, |T| <= 1/2, whose rows sum to at
// most 137 over all 189 offsets.  Two things make it cheap here:
//   * numbers of 59 and 57 bits as a high part and a signed low part of 30:
//     the product of the high parts and the two cross products are one
//     32 x 32 + 64-bit multiply-add each (exact sums; the product of the low
//     parts, below 2^-2 of the sums' last bit, is left out), ~15 cycles where
//     one FP64 multiply-add takes 64.  (Single-precision multiply-adds of the
//     low parts take half of that, but round at 2^-24 of sums that start at
//     2^-28 of the product: with the scales of mc_m2l_scale.cuh and a carry
//     every two columns the degrees above 4 still came out up to 2.4 times as
//     far from exact translations as in FP64, 8 times beside a dense cell);
//   * in the real layout a reflection x -> -x (y, z) only changes signs:
//     T_(s o) = X_s T_o X_s with X_s diagonal, +-1, so that the up to eight
//     offsets that differ in signs share one product:
//       sum_s T_(s o) M_s = sum_c T_o[r][c] Mt_d[c],  d = class(r) ^ class(c),
//       Mt_d = sum_s (-1)^(s . d) M_s
//     (class: the parities of a coefficient under the three reflections; Mt
//     a Walsh-Hadamard transform of eight cells' multipoles).  189 products
//     per cell become 56.
// A CTA takes 32 target cells of one parity class; warp k computes the rows of
// class k, so that all its products take their Mt from one transform index
// per column.  Half of the lanes take half of the rows, each lane two targets:
// a matrix entry and a transform value are loaded for several products each
// (one target per lane would return an entry to 32 lanes for each product).
// Level 6 of N = 1e6, p = 12 (32768 cells): 427 ms in FP64, 31 ms here, level
// 5 (4096 cells) 61 and 4.1; the multiply-adds alone would take 60 % of that,
// the rest are the transforms and the barriers between tiles.
#include <math.h>

#include <algorithm>

#include "mc_dev.cuh"
#include "mc_fix.cuh"
#include "mc_fixsum.cuh"
#include "mc_m2l.cuh"
#include "mc_m2l_scale.cuh"

namespace {

constexpr int kOrbits = 56;   // offsets up to signs: {0..3}^3 without {0, 1}^3
constexpr int kMaxRows = (MC_PMAX + 1) * (MC_PMAX + 1) + 32;
constexpr int kBitsT = 59, kBitsM = 57, kLimb = 30;

// Form of a CTA: 8 warps, two CTAs per SM, or, where 128 registers do not hold
// two targets' sums of half a class's rows, 16 warps of which two share a class's
// targets (fast setup of N = 1e6, p = 12: 42.5 ms; 8 warps with spills 51.5, with
// 240 registers and one CTA per SM 48.7)
__host__ __device__ __forceinline__ int warps_of(int p) { return p <= 11 ? 8 : 16; }
// columns staged at a time (one per warp), and tiles of the columns: at least
// two, so that an orbit's cells are known a step before its first tile is loaded
__host__ __device__ __forceinline__ int tiles_of(int p) {
  const int C = (p + 1) * (p + 1), tile = warps_of(p);
  return C <= tile ? 2 : (C + tile - 1) / tile;
}

// Rows by class; a class is two halves of `half` rows (the rows of the lower
// and upper 16 lanes), each padded to an even number.
struct M2LLayout {
  int start[8], half[8], rows;
  short index[kMaxRows];  // real-layout index of a row, -1: padding
};

// parities under x -> -x (bit 2), y -> -y (bit 1), z -> -z (bit 0)
int class_of(int n, int m, int im) { return (((m + im) & 1) << 2) | (im << 1) | ((n + m) & 1); }

M2LLayout m2l_layout(int p) {
  M2LLayout L;
  L.rows = 0;
  for (int c = 0; c < 8; c++) {
    short rows[kMaxRows];
    int cnt = 0;
    for (int n = 0; n <= p; n++)
      for (int m = 0; m <= n; m++)
        for (int im = 0; im < (m ? 2 : 1); im++)
          if (class_of(n, m, im) == c) rows[cnt++] = (short)(n * n + (m ? 2 * m - 1 : 0) + im);
    const int half = (cnt + 1) / 2, pad = (half + 1) / 2 * 2;
    L.start[c] = L.rows;
    L.half[c] = half;
    for (int i = 0; i < 2 * pad; i++) {
      const int r = (i / pad) * half + i % pad;
      L.index[L.rows++] = i % pad < half && r < cnt ? rows[r] : (short)-1;
    }
  }
  return L;
}

struct M2LArgs {
  int l, nl, h, pbc, p, nco, per_o;
  int start[8], half[8], rows;
  unsigned char ccol[kMaxRows];  // class of a column
  unsigned char orbit[kOrbits];  // |ox| | |oy| << 2 | |oz| << 4
  unsigned char degree[kMaxRows];  // of a row
  short index[kMaxRows];
  double scale[kMaxRows];
};

__device__ __forceinline__ void decode(int k, int* n, int* m, int* im) {
  int r = (int)sqrtf((float)k + 0.5f);
  while (r * r > k) r--;
  while ((r + 1) * (r + 1) <= k) r++;
  *n = r;
  const int rem = k - r * r;
  *m = (rem + 1) / 2;
  *im = (rem > 0 && (rem & 1) == 0) ? 1 : 0;
}

// h, l of v = h 2^30 + l, l signed
__device__ __forceinline__ int2 limbs(long long v) {
  const int l = ((int)v << (32 - kLimb)) >> (32 - kLimb);
  return make_int2((int)((v - l) >> kLimb), l);
}

struct TableArgs {
  int p, rows;
  signed char col[MC_PMAX + 1];
  unsigned char orbit[kOrbits];
  short index[kMaxRows];
};

// T_o[row][col] from the scaled irregular harmonics of the integer offsets
// (k_offset_table); entry (orbit, col, row)
__global__ void k_m2l_tables(const __grid_constant__ TableArgs A, const double* __restrict__ otab, int2* __restrict__ T) {
  const int p = A.p, C = (p + 1) * (p + 1), cpad = tiles_of(p) * warps_of(p);
  const int per = (2 * p + 1) * (2 * p + 2) / 2;
  const long long total = (long long)kOrbits * cpad * A.rows;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
    const int r = (int)(i % A.rows), col = (int)(i / A.rows % cpad), ob = A.orbit[i / A.rows / cpad];
    double v = 0.0;
    if (A.index[r] >= 0 && col < C) {
      int j, k, rim, n, m, cim;
      decode(A.index[r], &j, &k, &rim);
      decode(col, &n, &m, &cim);
      const double* t0 = otab + 2 * (size_t)((((ob & 3) + 3) * 7 + ((ob >> 2) & 3) + 3) * 7 + ((ob >> 4) & 3) + 3) * per;
      const int l = j + n;
      t0 += l * (l + 1);
      const int d = m - k, ad = d < 0 ? -d : d;
      const double sg = (min(k, m) & 1) ? -1.0 : 1.0;
      const double ar = sg * t0[2 * ad], ai = (d < 0 ? -sg : sg) * t0[2 * ad + 1];
      const double br = t0[2 * (m + k)], bi = t0[2 * (m + k) + 1];
      if (m == 0) {
        v = rim ? ai : ar;
      } else {
        v = rim ? (cim ? ar - br : ai - bi) : (cim ? -(ai + bi) : ar + br);
      }
      if (n & 1) v = -v;
      double f = 1.0, g = 1.0;
      for (int q = 2; q <= j - k; q++) f *= q;
      for (int q = 2; q <= j + k; q++) f *= q;
      for (int q = 2; q <= n - m; q++) g *= q;
      for (int q = 2; q <= n + m; q++) g *= q;
      v /= sqrt(f) * sqrt(g);
      v = ldexp(v, kBitsT + kM2LRowScale[m2l_group(ob)][j] - A.col[n]);
    }
    const long long w = __double2ll_rn(v);
    T[i] = limbs(w);
  }
}

struct ConvArgs {
  int nl, C;
  double scale[kMaxRows];  // sqrt((n-m)!(n+m)!) w^-n 2^kM2LColScale[n]
};

// one level's multipoles (scaled layout, by cell) as integers of kBitsM bits
// in units of a power of two per cell, stored by column; cells ordered by
// parity class, then by halved coordinates (consecutive lanes of a translation
// read consecutive cells)
__global__ void __launch_bounds__(256)
    k_m2l_convert(const __grid_constant__ ConvArgs A, const double* __restrict__ K, long long* __restrict__ M,
                  int* __restrict__ E) {
  extern __shared__ long long tile[];  // [32][C + 1]
  const int C = A.C, nl = A.nl, h = nl >> 1, h3 = h * h * h, ncl = nl * nl * nl;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, base = blockIdx.x * 32;
  for (int c = warp; c < 32; c += 8) {
    const int pos = base + c;
    if (pos >= ncl) break;
    const int cls = pos / h3, r = pos % h3;
    const int i = 2 * (r / (h * h)) + ((cls >> 2) & 1), j = 2 * ((r / h) % h) + ((cls >> 1) & 1), k = 2 * (r % h) + (cls & 1);
    const double* src = K + (size_t)((i * nl + j) * nl + k) * C;
    double v[8];
    int e = -4096;
#pragma unroll
    for (int u = 0; u < 8; u++) {
      const int col = lane + 32 * u;
      v[u] = col < C ? src[col] * A.scale[col] : 0.0;
      if (v[u] != 0.0) e = max(e, (int)((__double_as_longlong(v[u]) >> 52) & 0x7ff) - 1022);
    }
    e = __reduce_max_sync(0xffffffffu, e);
    if (lane == 0) E[pos] = e;
#pragma unroll
    for (int u = 0; u < 8; u++) {
      const int col = lane + 32 * u;
      if (col < C) tile[c * (C + 1) + col] = e == -4096 ? 0ll : __double2ll_rn(ldexp(v[u], kBitsM - e));
    }
  }
  __syncthreads();
  if (base + lane < ncl)
    for (int col = warp; col < C; col += 8) M[(size_t)col * ncl + base + lane] = tile[lane * (C + 1) + col];
}

// a b + c in one instruction (with the carry form of the sums over charges the
// fast setup of N = 1e6, p = 12 takes 49.5 instead of 42.5 ms)
__device__ __forceinline__ long long m2l_wide(int a, int b, long long c) {
  long long r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
}

template <int W>
__device__ __forceinline__ void cta_sync() {
  asm volatile("bar.sync 1, %0;" ::"n"(32 * W) : "memory");
}
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}

// warp w's class: the two warps of a sub-partition (w, w + 4) take opposite
// classes, whose rows add up to nearly a quarter of all (28 + 15 and 3 x 42 of
// 169 at p = 12)
__device__ __forceinline__ int class_of_warp(int w) { return w < 4 ? w : 11 - w; }

// 8 bytes, or zeros
__device__ __forceinline__ void cp_async8(void* dst, const void* src, bool valid) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  const int n = valid ? 8 : 0;
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(d), "l"(src), "r"(n) : "memory");
}

struct M2LShared {
  int2* T;        // [2][warps][rows]: table columns
  int2* Mt;       // [2][warps][8][32]: transform values
  long long* raw; // [warps][8][32]: the members' multipoles on their way there
  int* cell;      // [2][8][32]: members' cells of an orbit (-1: none), by lane
  int* shift;     // [2][8][32]: shifts to the unit of the orbit's group
  int* unit;      // [MC_M2L_GROUPS][32]: that unit (its exponent; -4096: no cell)
};

struct M2LTask {
  int cls, oc;  // target class, orbit chunk
  int I[3], b[3];  // the target this thread stages (clamped): halved coordinates, parities
  bool valid;
};

// halved coordinate and parity of coordinate 2 I + b + o on an axis with h
// halves (wrapped, or -1 outside)
__device__ __forceinline__ int half_of(int I, int b, int o, int h, bool pbc, int* par) {
  const int e = b + o;
  *par = e & 1;
  const int v = I + ((e - *par) >> 1);
  return pbc ? mc_wrap_coord(v, h) : (v < 0 || v >= h ? -1 : v);
}

// position (class-major) of the cell at offset o from this lane's target
__device__ __forceinline__ int cell_at(const M2LTask& k, int ox, int oy, int oz, int h, bool pbc) {
  int p0, p1, p2;
  const int a = half_of(k.I[0], k.b[0], ox, h, pbc, &p0), b = half_of(k.I[1], k.b[1], oy, h, pbc, &p1),
            c = half_of(k.I[2], k.b[2], oz, h, pbc, &p2);
  if (a < 0 || b < 0 || c < 0) return -1;
  return ((((p0 << 2 | p1 << 1 | p2) * h + a) * h) + b) * h + c;
}

// One CTA's task, as the warp that owns class w of NR rows sees it: every
// thread stages its target's part of the next tile's Mt and of the table
// columns while its warp computes the current ones.
template <int W, int NR>  // warps of the CTA, rows of half a class
__device__ __forceinline__ void m2l_task(const M2LArgs& A, const int2* __restrict__ T, const long long* __restrict__ M,
                                         const int* __restrict__ E, double* __restrict__ out, const M2LTask& k,
                                         const M2LShared& S, int t0, int w, int lane) {
  constexpr int NT = 16 / W, kTile = W;
  const int C = (A.p + 1) * (A.p + 1), tiles = (C + kTile - 1) / kTile > 1 ? (C + kTile - 1) / kTile : 2, h = A.h;
  const int ncl = A.nl * A.nl * A.nl;
  const int ob = k.oc * A.per_o, oe = min(kOrbits, ob + A.per_o);
  const int steps = (oe - ob) * tiles, tsz = kTile * A.rows;
  const int tid = 32 * w + lane, cls = class_of_warp(w & 7);
  const int tb = NT == 2 ? lane & 15 : (w >> 3) * 16 + (lane & 15);  // this lane's (first) target
  // products of the high parts, and the two cross products
  long long hh[NR > 0 ? NR : 1][NT], x[NR > 0 ? NR : 1][NT];
#pragma unroll
  for (int r = 0; r < NR; r++)
#pragma unroll
    for (int t = 0; t < NT; t++) hh[r][t] = x[r][t] = 0;
  int lo = ob, lt = 0;  // orbit and tile to load next
  // member w (signs of its offset: bits x 4, y 2, z 1) of an orbit
  auto members = [&](int o) {
    if (W > 8 && w >= 8) return;
    int of[3];
    bool ok = k.valid;
#pragma unroll
    for (int d = 0; d < 3; d++) {
      const int a = (A.orbit[o] >> (2 * d)) & 3, neg = (w >> (2 - d)) & 1;
      if ((a == 0 && neg) || (a == 3 && neg != k.b[d])) ok = false;
      of[d] = neg ? -a : a;
    }
    const int c = ok ? cell_at(k, of[0], of[1], of[2], h, A.pbc != 0) : -1;
    const int i = ((o & 1) * 8 + w) * 32 + lane;
    S.cell[i] = c;
    S.shift[i] = c >= 0 ? min(63, S.unit[m2l_group(A.orbit[o]) * 32 + lane] - E[c]) : 0;
  };
  // column w of the next tile: its lane's target's members, and the table
  auto load = [&](int s) {
    const int col = lt * kTile + w;
    const long long* Mc = M + (size_t)min(col, C - 1) * ncl;
    const int* cl = S.cell + (lo & 1) * 256 + lane;
#pragma unroll
    for (int g = 0; g < 8; g++) {
      const int c = cl[32 * g];
      cp_async8(&S.raw[(w * 8 + g) * 32 + lane], &Mc[max(c, 0)], c >= 0 && col < C);
    }
    const char* src = reinterpret_cast<const char*>(T + ((size_t)lo * tiles + lt) * tsz);
    char* dst = reinterpret_cast<char*>(S.T + (s & 1) * tsz);
    for (int i = 16 * tid; i < tsz * (int)sizeof(int2); i += 16 * 32 * W) cp_async16(dst + i, src + i);
    asm volatile("cp.async.commit_group;" ::: "memory");
    if (++lt == tiles) {
      lt = 0;
      lo++;
    } else if (lt == tiles - 1 && lo + 1 < oe) {
      members(lo + 1);  // read from the step after next on
    }
  };
  int so = ob, stl = 0;  // orbit and tile to transform next
  auto store = [&](int s) {
    // (each thread reads back what it copied itself)
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    int2* dst = S.Mt + (size_t)((s & 1) * kTile + w) * 8 * 32 + lane;
    const int* sh = S.shift + (so & 1) * 256 + lane;
    long long v[8];
#pragma unroll
    for (int g = 0; g < 8; g++) v[g] = S.raw[(w * 8 + g) * 32 + lane] >> sh[32 * g];
#pragma unroll
    for (int b = 1; b < 8; b <<= 1)
#pragma unroll
      for (int g = 0; g < 8; g++)
        if (!(g & b)) {
          const long long p = v[g], q = v[g | b];
          v[g] = p + q;
          v[g | b] = p - q;
        }
    // transform index d = (x, y, z) bits (4, 2, 1) of the member signs
#pragma unroll
    for (int d = 0; d < 8; d++) dst[d * 32] = limbs(v[d]);
    if (++stl == tiles) {
      stl = 0;
      so++;
    }
  };
  // a group's sums into the result
  bool first = true;
  auto flush = [&](int g) {
    const int h3 = h * h * h;
#pragma unroll
    for (int t = 0; t < NT; t++) {
      const int ii = t0 + 16 * t + tb;
      const double unit = ldexp(1.0, S.unit[g * 32 + 16 * t + tb]);
      const int i = 2 * (ii / (h * h)) + k.b[0], j = 2 * ((ii / h) % h) + k.b[1], kk = 2 * (ii % h) + k.b[2];
      double* o = out + ((size_t)((i * A.nl + j) * A.nl + kk) * A.nco + k.oc) * C;
#pragma unroll
      for (int r = 0; r < NR; r++) {
        const int row = A.start[cls] + (lane >> 4) * ((NR + 1) / 2 * 2) + r, at = A.index[row];
        if (ii < h3 && at >= 0) {
          const double down = __longlong_as_double((long long)(1023 - kM2LRowScale[g][A.degree[row]]) << 52);
          const double v = fma((double)x[r][t], 1.0 / (double)(1 << kLimb), (double)hh[r][t]) * A.scale[row] * down * unit;
          o[at] = first ? v : o[at] + v;
        }
        hh[r][t] = x[r][t] = 0;
      }
    }
    first = false;
  };
  members(ob);
  cta_sync<W>();
  load(0);
  store(0);
  cta_sync<W>();
  int tile = 0, co = ob;  // of the current step: tile and orbit
  for (int s = 0; s < steps; s++) {
    if (s + 1 < steps) load(s + 1);
    if constexpr (NR > 0) {
      const int2* tt = S.T + (s & 1) * tsz + A.start[cls] + (lane >> 4) * ((NR + 1) / 2 * 2);
      const int2* m0 = S.Mt + (size_t)(s & 1) * kTile * 8 * 32 + tb;
#pragma unroll 1
      for (int c0 = 0; c0 < kTile; c0 += 8) {
#pragma unroll 2
        for (int c = c0; c < c0 + 8; c++) {
          const int d = cls ^ A.ccol[tile * kTile + c];
          int2 m[NT];
#pragma unroll
          for (int t = 0; t < NT; t++) m[t] = m0[(c * 8 + d) * 32 + 16 * t];
          const int4* tr = reinterpret_cast<const int4*>(tt + c * A.rows);
#pragma unroll
          for (int r = 0; r < NR; r++) {
            const int4 q = tr[r / 2];
            const int th = r & 1 ? q.z : q.x, tl = r & 1 ? q.w : q.y;
#pragma unroll
            for (int t = 0; t < NT; t++) {
              hh[r][t] = m2l_wide(th, m[t].x, hh[r][t]);
              x[r][t] = m2l_wide(th, m[t].y, x[r][t]);
              x[r][t] = m2l_wide(tl, m[t].x, x[r][t]);
            }
          }
        }
        // |x| < 8 (2^29 2^29 + 2^29 2^30) + 2^30 < 2^63 between two carries
        static_assert(kBitsT - kLimb <= 29 && kBitsM + 3 - kLimb <= 30 && kLimb <= 30, "cross products");
#pragma unroll
        for (int r = 0; r < NR; r++)
#pragma unroll
          for (int t = 0; t < NT; t++) {
            hh[r][t] += x[r][t] >> kLimb;
            x[r][t] &= (1 << kLimb) - 1;
          }
      }
    }
    if (++tile == tiles) {
      tile = 0;
      const int g = m2l_group(A.orbit[co]);
      if (++co == oe || m2l_group(A.orbit[co]) != g) flush(g);
    }
    if (s + 1 < steps) store(s + 1);
    cta_sync<W>();
  }
}

}  // namespace

template <int W>
__global__ void __launch_bounds__(32 * W, 16 / W)
    k_m2l_fix(const __grid_constant__ M2LArgs A, const int2* __restrict__ T, const long long* __restrict__ M,
              const int* __restrict__ E, double* __restrict__ out) {
  extern __shared__ int4 dyn4[];
  constexpr int kTargets = 32;
  M2LShared S;
  S.T = reinterpret_cast<int2*>(dyn4);
  S.Mt = S.T + 2 * W * A.rows;
  S.raw = reinterpret_cast<long long*>(S.Mt + 2 * W * 8 * 32);
  S.cell = reinterpret_cast<int*>(S.raw + W * 8 * 32);
  S.shift = S.cell + 2 * 8 * 32;
  S.unit = S.shift + 2 * 8 * 32;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int h = A.h, h3 = h * h * h, chunks = (h3 + kTargets - 1) / kTargets;
  M2LTask k;
  k.oc = blockIdx.x % A.nco;
  const int tk = blockIdx.x / A.nco;
  k.cls = tk / chunks;
  const int t0 = (tk % chunks) * kTargets, ii = t0 + threadIdx.x % kTargets;
  k.valid = ii < h3;
  const int r = min(ii, h3 - 1);
  k.I[0] = r / (h * h);
  k.I[1] = (r / h) % h;
  k.I[2] = r % h;
#pragma unroll
  for (int d = 0; d < 3; d++) k.b[d] = (k.cls >> (2 - d)) & 1;
  // units of the sums: the largest of the cells at a group's offsets
  static_assert(kTargets == 32, "a target per lane");
  for (int i = threadIdx.x; i < MC_M2L_GROUPS * 32; i += 32 * W) S.unit[i] = -4096;
  __syncthreads();
  for (int q = w; q < 216; q += W) {
    const int ox = q / 36 - 2 - k.b[0], oy = (q / 6) % 6 - 2 - k.b[1], oz = q % 6 - 2 - k.b[2];
    if (ox >= -1 && ox <= 1 && oy >= -1 && oy <= 1 && oz >= -1 && oz <= 1) continue;
    const int c = cell_at(k, ox, oy, oz, h, A.pbc != 0);
    if (c >= 0 && k.valid) atomicMax(&S.unit[m2l_group(abs(ox) | abs(oy) << 2 | abs(oz) << 4) * 32 + lane], E[c]);
  }
  __syncthreads();
  // half of 1, 3, 6, 10, 15, 21, 28, 36 rows
#define MC_M2L_ROWS(NR_) \
  case NR_: m2l_task<W, NR_>(A, T, M, E, out, k, S, t0, w, lane); break;
  switch (A.half[class_of_warp(w & 7)]) {
    MC_M2L_ROWS(1)
    MC_M2L_ROWS(2)
    MC_M2L_ROWS(3)
    MC_M2L_ROWS(5)
    MC_M2L_ROWS(8)
    MC_M2L_ROWS(11)
    default:
      // (0 rows; any other number would leave its results out, but no barrier)
      if constexpr (W == 16) {
        switch (A.half[class_of_warp(w & 7)]) {
          MC_M2L_ROWS(14)
          MC_M2L_ROWS(18)
          default: m2l_task<W, 0>(A, T, M, E, out, k, S, t0, w, lane);
        }
      } else {
        m2l_task<W, 0>(A, T, M, E, out, k, S, t0, w, lane);
      }
  }
#undef MC_M2L_ROWS
}

__global__ void k_offset_table(int p, double* __restrict__ out);

size_t m2l_table_bytes(int p) {
  return sizeof(int2) * (size_t)kOrbits * tiles_of(p) * warps_of(p) * m2l_layout(p).rows;
}

// by group
static void orbits(unsigned char* o) {
  int n = 0;
  for (int g = 0; g < MC_M2L_GROUPS; g++)
    for (int i = 0; i < 64; i++)
      if (((i & 3) > 1 || ((i >> 2) & 3) > 1 || i >> 4 > 1) && m2l_group(i) == g) o[n++] = (unsigned char)i;
}

cudaError_t m2l_build_table(int p, int sms, void* table, double* otab, cudaStream_t st) {
  const int per = (2 * p + 1) * (2 * p + 2) / 2;
  k_offset_table<<<std::max(1, std::min(sms * 8, (343 * per + 255) / 256)), 256, 0, st>>>(p, otab);
  TableArgs A;
  const M2LLayout L = m2l_layout(p);
  A.p = p;
  A.rows = L.rows;
  std::copy(kM2LColScale, kM2LColScale + MC_PMAX + 1, A.col);
  std::copy(L.index, L.index + L.rows, A.index);
  orbits(A.orbit);
  k_m2l_tables<<<sms * 8, 256, 0, st>>>(A, otab, (int2*)table);
  return cudaGetLastError();
}

static double sfac(int n, int m) {
  double f = 1.0, g = 1.0;
  for (int q = 2; q <= n - m; q++) f *= q;
  for (int q = 2; q <= n + m; q++) g *= q;
  return sqrt(f) * sqrt(g);
}

int m2l_chunks(int nl, int sms) {
  const int h = nl / 2, tasks = 8 * ((h * h * h + 31) / 32);
  // at least twelve tasks per SM (two at a time), so that the last wave is short
  return std::max(1, std::min(kOrbits, (12 * sms + tasks - 1) / tasks));
}

cudaError_t m2l_fix_level(int p, int l, double w, bool pbc, int sms, const void* table, const double* K, long long* M,
                          int* E, double* Lout, double* scratch, size_t scratch_doubles, cudaStream_t st) {
  const int C = (p + 1) * (p + 1), nl = 1 << (l - 1), h = nl / 2, ncl = nl * nl * nl;
  const M2LLayout L = m2l_layout(p);
  ConvArgs V;
  V.nl = nl;
  V.C = C;
  M2LArgs A;
  A.l = l;
  A.nl = nl;
  A.h = h;
  A.pbc = pbc;
  A.p = p;
  A.nco = m2l_chunks(nl, sms);
  while (A.nco > 1 && (size_t)ncl * A.nco * C > scratch_doubles) A.nco--;
  A.per_o = (kOrbits + A.nco - 1) / A.nco;
  A.nco = (kOrbits + A.per_o - 1) / A.per_o;
  A.rows = L.rows;
  for (int c = 0; c < 8; c++) {
    A.start[c] = L.start[c];
    A.half[c] = L.half[c];
  }
  orbits(A.orbit);
  std::fill(A.ccol, A.ccol + kMaxRows, 0);
  for (int n = 0; n <= p; n++) {
    const double wn = pow(w, -(double)n);
    for (int m = 0; m <= n; m++)
      for (int im = 0; im < (m ? 2 : 1); im++) {
        const int k = n * n + (m ? 2 * m - 1 : 0) + im;
        A.ccol[k] = (unsigned char)class_of(n, m, im);
        V.scale[k] = sfac(n, m) * wn * (double)(1 << kM2LColScale[n]);
      }
  }
  for (int r = 0; r < L.rows; r++) {
    A.index[r] = L.index[r];
    A.scale[r] = 0.0;
    A.degree[r] = 0;
    if (L.index[r] < 0) continue;
    int n = (int)sqrt((double)L.index[r] + 0.5);
    const int rem = L.index[r] - n * n, m = (rem + 1) / 2;
    A.degree[r] = (unsigned char)n;
    A.scale[r] = sfac(n, m) * pow(w, -(double)(n + 1)) * ldexp(1.0, 2 * kLimb - kBitsT - kBitsM);
  }
  const size_t csm = sizeof(long long) * 32 * (C + 1);
  cudaError_t e = cudaFuncSetAttribute(k_m2l_convert, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)csm);
  if (e != cudaSuccess) return e;
  k_m2l_convert<<<(ncl + 31) / 32, 256, csm, st>>>(V, K, M, E);
  const int chunks = (h * h * h + 31) / 32;
  const int warps = warps_of(p);
  const size_t smem = sizeof(int2) * (2 * (size_t)warps * L.rows + 3 * warps * 8 * 32) + sizeof(int) * (4 * 8 + MC_M2L_GROUPS) * 32;
  const auto kernel = warps == 8 ? k_m2l_fix<8> : k_m2l_fix<16>;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  kernel<<<8 * chunks * A.nco, 32 * warps, smem, st>>>(A, (const int2*)table, M, E, A.nco > 1 ? scratch : Lout);
  e = cudaGetLastError();
  if (e == cudaSuccess && A.nco > 1) e = fix_reduce(ncl, A.nco, C, sms, scratch, Lout, st);
  return e;
}
