// Harmonic sums over charges in 64-bit fixed point on the integer pipe:
//   irregular  S_n^m = sum_i q_i conj It_n^m(r_i - R)   (Alg. L.3)
//   regular    S_n^m = sum_i q_i conj Rt_n^m(r_i - R)   (Eq. 4)
// GB300 issues one FP64 warp instruction per ~64 cycles and sub-partition,
// but a 32 x 32 + 64 bit integer multiply-add every ~4.3 cycles (both
// measured), so a 62-bit product of three or four multiply-adds costs 13 to 17
// cycles against 64 for one FP64 instruction, and it keeps more bits: every
// quantity below is bounded by 1 by construction, is held to 2^-59 .. 2^-63,
// and is summed exactly.
//
// Scaling.  With R0 a radius every source satisfies (r >= R0 irregular,
// r <= R0 regular), rho = R0/r (or r/R0) <= 1, zeta = rho cos t,
// kappa = rho^2 and F_n^m = P_n^m / sin^m t / (its value at the pole),
//   It_n^m = (n+m)! / (2^m m!) R0^-(n+1) e^{i m phi} Y,  Y = rho (rho sin t)^m rho^(n-m) F_n^m(cos t)
//   Rt_n^m = R0^n / (2^m m! (n-m)!)      e^{i m phi} Y   (Y without the first rho).
// q Y, kept within 1 by a power of two close to its normalisation
// sqrt((n-m)!/(n+m)!) (n+m)!/(2^m m!) (|Y_n^m| <= 1, so no bit is lost
// where the value at the pole is hundreds of times larger), obeys
//   Y_n = 2^tau_n (zeta Y_{n-1} - w_n kappa Y_{n-2}),  Y_m = q rho (rho sin t)^m.
// Signs s_n = +, +, -, - (period 4 in n - m) turn the difference into
// Y_n = 2^tau_n (+-zeta Y_{n-1} + w_n kappa Y_{n-2}) without negations.
//
// Needs only <stdint.h>, an inverse square root and the qualifiers below, so
// it also compiles for host tests.
#pragma once
#include <math.h>
#include <stdint.h>

#ifndef MC_PMAX
#define MC_PMAX 15
#endif
#define MC_FIX_WARPS 4   // warps that share the columns
#define MC_FIX_STEPS 34  // most recurrence steps of one warp (p = 15)
// groups of 32 charges between two flushes of a lane's sums: one term is at
// most 2^58, so 28 stay below 2^63, and halved before each exchange the sum
// over the 32 lanes does too (a bit more for the terms would double the
// flushes, 3 % of the kernel)
#define MC_FIX_FLUSH 28
#define MC_FIX_PHASE 2  // cos m phi, sin m phi enter the terms as multiples of 2^-60

// value h 2^32 + l with signed l, so that every partial product is a signed
// 32 x 32 one
struct Fx {
  int32_t h, l;
};
__host__ __device__ __forceinline__ Fx fx_split(int64_t v) {
  Fx r;
  r.l = (int32_t)v;
  r.h = (int32_t)((uint32_t)((uint64_t)v >> 32) + ((uint32_t)v >> 31));
  return r;
}
// a b + c as two multiply-adds with a carry between them.  The one wide
// instruction takes the same 4.3 cycles but wants its sum in an aligned
// register pair: with it Alg. L.3 for 1e5 charges at L = 4 took 5.35 instead
// of 4.74 ms (the C expressions cost half as much again)
__host__ __device__ __forceinline__ int64_t fx_wide(int32_t a, int32_t b, int64_t c) {
#ifdef __CUDA_ARCH__
  int32_t lo = (int32_t)c, hi = (int32_t)(c >> 32);
  asm("mad.lo.cc.s32 %0, %2, %3, %0;\n\tmadc.hi.s32 %1, %2, %3, %1;" : "+r"(lo), "+r"(hi) : "r"(a), "r"(b));
  return (int64_t)(((uint64_t)(uint32_t)hi << 32) | (uint32_t)lo);
#else
  return (int64_t)((uint64_t)((int64_t)a * (int64_t)b) + (uint64_t)c);
#endif
}
__host__ __device__ __forceinline__ uint64_t fx_wideu(uint32_t a, uint32_t b, uint64_t c) {
#ifdef __CUDA_ARCH__
  uint32_t lo = (uint32_t)c, hi = (uint32_t)(c >> 32);
  asm("mad.lo.cc.u32 %0, %2, %3, %0;\n\tmadc.hi.u32 %1, %2, %3, %1;" : "+r"(lo), "+r"(hi) : "r"(a), "r"(b));
  return ((uint64_t)hi << 32) | lo;
#else
  return (uint64_t)a * (uint64_t)b + c;
#endif
}
constexpr int64_t kFxHalf = 0x80000000LL;

// (r + (low half of t) / 2^32) 2^s, s < 32, for a cross product t whose high
// half is in r already: the bits below r's last one come from t (a plain shift would fill zeros in: the
// values would be good to 2^-59 instead of 2^-61)
__host__ __device__ __forceinline__ int64_t fx_shl(int64_t t, int64_t r, int s) {
#ifdef __CUDA_ARCH__
  const uint32_t lo = __funnelshift_l((uint32_t)t, (uint32_t)r, s);
  const uint32_t hi = __funnelshift_l((uint32_t)r, (uint32_t)((uint64_t)r >> 32), s);
  return (int64_t)(((uint64_t)hi << 32) | lo);
#else
  return (int64_t)(((uint64_t)r << s) | ((uint64_t)(uint32_t)t >> (32 - s)));
#endif
}
// a b / 2^(64 - s), 0 < s < 32; the product of the low parts (below 2^-2 of
// the last bit before the shift) left out
__host__ __device__ __forceinline__ int64_t fx_mul(Fx a, Fx b, int s) {
  const int64_t t = fx_wide(a.h, b.l, fx_wide(a.l, b.h, 0));
  return fx_shl(t, fx_wide(a.h, b.h, t >> 32), s);
}
// a b / 2^32 for a 31-bit a
__host__ __device__ __forceinline__ int64_t fx_mulint(int32_t a, Fx b) {
  return fx_wide(a, b.h, fx_wide(a, b.l, kFxHalf) >> 32);
}
// a b / 2^62, and a c - b d, a d + b c over 2^62: one step of the powers of
// st and of e^{i phi}
__host__ __device__ __forceinline__ int64_t fx_mul62(Fx a, Fx b) {
  return fx_mul(a, b, 2);
}
__host__ __device__ __forceinline__ void fx_turn(Fx a, Fx b, Fx c, Fx d, Fx dn, int64_t* re, int64_t* im) {
  int64_t t = fx_wide(a.l, c.h, 0), u = fx_wide(a.l, d.h, 0);
  t = fx_wide(a.h, c.l, t);
  u = fx_wide(a.h, d.l, u);
  t = fx_wide(b.l, dn.h, t);
  u = fx_wide(b.l, c.h, u);
  t = fx_wide(b.h, dn.l, t);
  u = fx_wide(b.h, c.l, u);
  const int64_t r = fx_wide(b.h, dn.h, fx_wide(a.h, c.h, t >> 32)), i = fx_wide(b.h, c.h, fx_wide(a.h, d.h, u >> 32));
  *re = fx_shl(t, r, 2);
  *im = fx_shl(u, i, 2);
}

// x / a in units of 2^-62 for 0 <= x <= a (1 + 2^-14): rcp = 2^115 / (mantissa
// of a), ea the biased exponent of a.  A row just beyond the upper face may
// have the next exponent (s = -1, where a is just below a power of two).
__host__ __device__ __forceinline__ int64_t fx_coord(double x, uint64_t rcp, int ea) {
#ifdef __CUDA_ARCH__
  const uint64_t u = (uint64_t)__double_as_longlong(x);
#else
  uint64_t u;
  __builtin_memcpy(&u, &x, 8);
#endif
  const int e = (int)((u >> 52) & 0x7ff);
  const int s = ea - e;
  if (e == 0 || s > 62) return 0;
  const uint64_t m = ((u & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull) << 11;
#ifdef __CUDA_ARCH__
  const uint64_t v = __umul64hi(m, rcp);
#else
  const uint64_t v = (uint64_t)(((unsigned __int128)m * rcp) >> 64);
#endif
  return (int64_t)(s < 0 ? v << 1 : v >> s);
}
// x in units of 2^-60 finest cells (2^62: four of them) modulo 2^64, for
// 0 <= x < a and L levels: r1 2^64 + r0 = 2^179 / (mantissa of a).  Rounded
// down by less than two units wherever x lies; a fraction of the box in 62
// bits, shifted up, was off by up to 2^(L-3) units.
__host__ __device__ __forceinline__ int64_t fx_cells(double x, uint64_t r1, uint64_t r0, int ea, int L) {
#ifdef __CUDA_ARCH__
  const uint64_t u = (uint64_t)__double_as_longlong(x);
#else
  uint64_t u;
  __builtin_memcpy(&u, &x, 8);
#endif
  const int e = (int)((u >> 52) & 0x7ff), s = ea - e - (L - 3);
  if (e == 0 || s > 62) return 0;
  const uint64_t m = ((u & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull) << 11;
#ifdef __CUDA_ARCH__
  const uint64_t h = __umul64hi(m, r1), l = __umul64hi(m, r0);
#else
  const uint64_t h = (uint64_t)(((unsigned __int128)m * r1) >> 64);
  const uint64_t l = (uint64_t)(((unsigned __int128)m * r0) >> 64);
#endif
  const uint64_t lo = m * r1 + l, hi = h + (lo < l);
  return (int64_t)(s > 0 ? hi >> s : s == 0 ? hi : (hi << -s) | (lo >> (64 + s)));
}
// q / 2^E in units of 2^-62 for |q| <= 2^E (E biased by 1023 like an exponent)
__host__ __device__ __forceinline__ int64_t fx_charge(double q, int Eb) {
#ifdef __CUDA_ARCH__
  const uint64_t u = (uint64_t)__double_as_longlong(q);
#else
  uint64_t u;
  __builtin_memcpy(&u, &q, 8);
#endif
  const int e = (int)((u >> 52) & 0x7ff);
  const int s = Eb - e;
  if (e == 0 || s > 62) return 0;
  const int64_t m = (int64_t)(((u & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull) << 10);
  const int64_t v = m >> s;
  return (u >> 63) ? -v : v;
}

// irregular sets: R0 = 1.5 cell widths (1 - 2^-12), below the distance 1.5 w
// of a target's centre from any charge of its interaction list; in units of
// four cell widths r0 = 0.375 (1 - 2^-12) = 12285 / 2^15
constexpr double kFixR0 = 1.5 * (1.0 - 1.0 / 4096.0);
constexpr uint64_t kFixC80 = (uint64_t)12285ull * 12285ull << 50;  // r0^2 2^80 mod 2^64
constexpr int64_t kFixCinv = (int64_t)(((unsigned __int128)1 << 90) / (12285ull * 12285ull));  // 2^60 / r0^2
constexpr int64_t kFixR0inv = (int64_t)(((unsigned __int128)1 << 76) / 12285ull);              // 2^61 / r0

// What the recurrence needs of one charge: zeta, e^{i phi} (ex, ey),
// st = rho sin t, x0 = Y_0 (all 2^62), kappa (2^63).  ex, ey may be longer
// than 1 by 2^-21 as long as st (ex, ey) = (x, y) rho/r, which is exact.
struct FixCharge {
  int64_t zeta, ex, ey, st, x0;
  uint64_t kap;
};

__host__ __device__ __forceinline__ int fx_clz(uint64_t v) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)v);
#else
  return __builtin_clzll(v);
#endif
}
__host__ __device__ __forceinline__ float fx_rsqrt(float v) {
#ifdef __CUDA_ARCH__
  return rsqrtf(v);
#else
  return 1.0f / __builtin_sqrtf(v);
#endif
}
__host__ __device__ __forceinline__ float fx_rcp(float v) {
#ifdef __CUDA_ARCH__
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
  return r;
#else
  return 1.0f / v;
#endif
}
// the sum of squares of two or three values of 2^62 in units of 2^-60
__host__ __device__ __forceinline__ int64_t fx_norm(Fx x, Fx y, Fx z) {
  int64_t t = fx_wide(x.h, x.l, (int64_t)1 << 30);
  t = fx_wide(y.h, y.l, t);
  t = fx_wide(z.h, z.l, t);
  return fx_wide(x.h, x.h, fx_wide(y.h, y.h, fx_wide(z.h, z.h, t >> 31)));
}

// (dx, dy) as s (ex, ey): the length of a 24-bit reciprocal root times its
// 62-bit reciprocal, taken after both are shifted up to full length
__host__ __device__ __forceinline__ int64_t fix_polar(int64_t dx, int64_t dy, FixCharge* f) {
  const uint64_t m = (uint64_t)(dx < 0 ? -dx : dx) | (uint64_t)(dy < 0 ? -dy : dy);
  if (m == 0) {
    f->ex = (int64_t)1 << 62;
    f->ey = 0;
    return 0;
  }
  const int k = fx_clz(m) - 2;
  const int64_t x = (int64_t)((uint64_t)dx << k), y = (int64_t)((uint64_t)dy << k);
  const int64_t n2 = fx_norm(fx_split(x), fx_split(y), Fx{0, 0});  // 1/4 .. 2
  const float rs = fx_rsqrt((float)(int32_t)(n2 >> 32) * 3.7252902984619140625e-9f);
  const int32_t ri = (int32_t)(rs * 536870912.0f);         // 2^29
  const int32_t s0 = (int32_t)(fx_rcp(rs) * 536870912.0f);  // 2^29
  // 1/rs = s0 (1 + e + e^2), e = 1 - rs s0 below 2^-20 (2^58)
  const int64_t e = ((int64_t)1 << 58) - (int64_t)ri * s0;
  const int32_t eh = (int32_t)(e >> 13);  // 2^45
  const int64_t c = e + (((int64_t)eh * eh) >> 32);
  const int64_t s = ((int64_t)s0 << 33) + (fx_mulint(s0, fx_split((int64_t)((uint64_t)c << 7))) >> 0);
  f->ex = (int64_t)((uint64_t)fx_mulint(ri, fx_split(x)) << 3);
  f->ey = (int64_t)((uint64_t)fx_mulint(ri, fx_split(y)) << 3);
  return k > 0 ? (s + ((int64_t)1 << (k - 1))) >> k : s;
}

// irregular: displacement (2^62 = four cell widths), charge q (2^62)
__host__ __device__ __forceinline__ FixCharge fix_irregular(int64_t dx, int64_t dy, int64_t dz, int64_t q) {
  const int64_t r2 = fx_norm(fx_split(dx), fx_split(dy), fx_split(dz));
  // rho from a single-precision estimate (relative error below 2^-20) and one
  // third-order step: rho (1 + e/2 + 3 e^2/8), e = 1 - rho^2 r^2 / r0^2
  const float yf = 0.374908447265625f * fx_rsqrt((float)(int32_t)(r2 >> 32) * 3.7252902984619140625e-9f);
  const int32_t yi = (int32_t)(yf * 1073741824.0f);
  const uint64_t y2 = (uint64_t)((int64_t)yi * yi);
  const uint64_t plo = y2 * (uint64_t)r2;
#ifdef __CUDA_ARCH__
  const uint64_t phi = __umul64hi(y2, (uint64_t)r2);
#else
  const uint64_t phi = (uint64_t)(((unsigned __int128)y2 * (uint64_t)r2) >> 64);
#endif
  const int64_t d = (int64_t)(kFixC80 - ((phi << 24) | (plo >> 40)));  // e r0^2 2^80
  const int64_t e = fx_mul(fx_split(d), fx_split(kFixCinv), 4);  // 2^80, below 2^60
  const int32_t eh = (int32_t)(e >> 32);
  const int64_t c = (e >> 1) + ((3 * (((int64_t)eh * eh) >> 16)) >> 3);
  const int64_t rho = ((int64_t)yi << 32) + (fx_mulint(yi, fx_split(c)) >> 16);
  FixCharge f;
  const Fx rs = fx_split(rho);
  f.kap = (uint64_t)fx_mul(rs, rs, 3);
  const Fx g = fx_split(fx_mul(fx_split((int64_t)(f.kap >> 1)), fx_split(kFixR0inv), 2));  // kappa / r0 (2^61)
  f.zeta = fx_mul(fx_split(dz), g, 3);
  f.st = fx_mul(fx_split(fix_polar(dx, dy, &f)), g, 3);
  f.x0 = fx_mul62(fx_split(q), rs);
  return f;
}
// regular: displacement (2^62 = one cell width = R0), charge q (2^62)
__host__ __device__ __forceinline__ FixCharge fix_regular(int64_t dx, int64_t dy, int64_t dz, int64_t q) {
  FixCharge f;
  f.kap = (uint64_t)fx_norm(fx_split(dx), fx_split(dy), fx_split(dz)) << 3;
  f.zeta = dz;
  f.st = fix_polar(dx, dy, &f);
  f.x0 = q;
  return f;
}

// One step of the recurrence.  zs = +-zeta, q1, q2 the two previous values,
// w = w_n (2^63), sh = 2 + tau_n.
__host__ __device__ __forceinline__ Fx fix_next(Fx zs, uint32_t kh, uint32_t kl, Fx q1, Fx q2, uint32_t wh,
                                                uint32_t wl, int sh) {
  // kappa w (2^62): both below 2^63, so the unsigned cross sum fits
  uint64_t s = fx_wideu(kl, wh, 0x80000000ull);
  s = fx_wideu(kh, wl, s);
#ifdef __CUDA_ARCH__
  uint64_t kw = fx_wideu(kh, wh, 0);
  asm("mad.wide.u32 %0, %1, 1, %0;" : "+l"(kw) : "r"((uint32_t)(s >> 32)));
#else
  const uint64_t kw = fx_wideu(kh, wh, s >> 32);
#endif
  const Fx k = fx_split((int64_t)kw);
  int64_t t = fx_wide(zs.l, q1.h, 0);
  t = fx_wide(zs.h, q1.l, t);
  t = fx_wide(k.l, q2.h, t);
  t = fx_wide(k.h, q2.l, t);
  int64_t r = fx_wide(zs.h, q1.h, t >> 32);
  r = fx_wide(k.h, q2.h, r);
  return fx_split(fx_shl(t, r, sh));
}
// acc + x y (phase x 2^60, y 2^62: terms of 2^58)
__host__ __device__ __forceinline__ int64_t fix_mac(Fx x, Fx q, int64_t acc) {
  int64_t t = fx_wide(x.l, q.h, kFxHalf);
  t = fx_wide(x.h, q.l, t);
  return acc + fx_wide(x.h, q.h, t >> 32);
}

// Steps of the longest of four shares of the columns m = 0..p (p - m + 1
// steps each): the smallest capacity that first-fit packing of the columns
// into four warps meets.  91 of 92 warp steps are used at p = 12.
struct FixShares {
  int steps;
  int warp[MC_PMAX + 1], first[MC_PMAX + 1];  // warp of column m, its first step there
};
constexpr FixShares fix_shares(int p) {
  for (int cap = p + 1;; cap++) {
    FixShares s{};
    int used[MC_FIX_WARPS] = {0, 0, 0, 0};
    bool ok = true;
    for (int m = 0; m <= p && ok; m++) {
      const int len = p - m + 1;
      int b = 0;
      while (b < MC_FIX_WARPS && used[b] + len > cap) b++;
      if (b == MC_FIX_WARPS) {
        ok = false;
      } else {
        s.warp[m] = b;
        s.first[m] = used[b];
        used[b] += len;
      }
    }
    if (ok) {
      s.steps = cap;
      return s;
    }
  }
}

// Tables of one launch: per warp and step the recurrence constants and the
// value of the step's sum in the scaled layout (times 2^-53); unused steps
// have scale 0 and index -1.
struct FixStep {
  uint32_t wh, wl;
  int32_t sh;
  int32_t pad;
};
struct FixTab {
  FixStep step[MC_FIX_WARPS][MC_FIX_STEPS];
  double scale[MC_FIX_WARPS][MC_FIX_STEPS];
  short index[MC_FIX_WARPS][MC_FIX_STEPS];      // of the real part in the real layout
  unsigned long long turn[MC_FIX_WARPS];        // steps where a column begins
  unsigned char col[MC_FIX_WARPS][MC_PMAX + 1]; // the warp's columns in order
};

// R: the radius R0 in length units; `unit` (optional) receives the scales for a
// radius of 1 before they are rounded
inline void fix_tab_build(FixTab* T, int p, bool irregular, double R, long double (*unit)[MC_FIX_STEPS] = nullptr) {
  const FixShares sh = fix_shares(p);
  int ncol[MC_FIX_WARPS] = {0, 0, 0, 0};
  for (int k = 0; k < MC_FIX_WARPS; k++) {
    T->turn[k] = 0;
    for (int m = 0; m <= MC_PMAX; m++) T->col[k][m] = 0;
    for (int t = 0; t < MC_FIX_STEPS; t++) {
      T->step[k][t] = FixStep{0u, 0u, 2, 0};
      T->scale[k][t] = 0.0;
      T->index[k][t] = -1;
    }
  }
  for (int m = 0; m <= p; m++) {
    const int k = sh.warp[m];
    T->turn[k] |= 1ull << sh.first[m];
    T->col[k][ncol[k]++] = (unsigned char)m;
    // prod: product of alpha (F = prod x monic); norm: normalisation of
    // monic e^{i m phi}, at most 1 over its largest value
    long double prod = 1.0L, aprev = 1.0L, norm = 1.0L;
    for (int i = 1; i <= m; i++) norm *= sqrtl((2.0L * i - 1.0L) / (2.0L * i));
    int sigma = 0, tau_prev = 0;
    long double head = 1.0L;  // (2m)!/(2^m m!) or 1/(2^m m!)
    for (int i = 1; i <= m; i++) head *= irregular ? (long double)(2 * i - 1) : 1.0L / (2.0L * i);
    long double rad = 1.0L;
    for (int i = 0; i < (irregular ? m + 1 : m); i++) rad *= irregular ? 1.0L / (long double)R : (long double)R;
    for (int n = m; n <= p; n++) {
      const int i = n - m, t = sh.first[m] + i;
      if (i > 0) {
        const long double alpha = (2.0L * n - 1.0L) / (n + m), beta = (n - m - 1.0L) / (n + m);
        prod *= alpha;
        norm *= (2.0L * n - 1.0L) / sqrtl((long double)(n - m) * (n + m));
        int sg = sigma;
        while (norm >= (long double)(2ull << sg)) sg++;
        const long double W = beta / (alpha * aprev) * (long double)(1 << tau_prev);
        const uint64_t w = (uint64_t)(W * 9223372036854775808.0L + 0.5L);
        T->step[k][t].wh = (uint32_t)(w >> 32);
        T->step[k][t].wl = (uint32_t)w;
        T->step[k][t].sh = 2 + sg - sigma;
        aprev = alpha;
        tau_prev = sg - sigma;
        sigma = sg;
        if (irregular) {
          head *= (long double)(n + m);
          rad /= (long double)R;
        } else {
          head /= (long double)(n - m);
          rad *= (long double)R;
        }
      }
      const long double sign = (i & 2) ? -1.0L : 1.0L;
      const long double one = head * sign * prod / (long double)(1ull << sigma) / 9007199254740992.0L;
      if (unit) unit[k][t] = one;
      T->scale[k][t] = (double)(one * rad);
      T->index[k][t] = (short)(n * n + (m ? 2 * m - 1 : 0));
    }
  }
}

// Near pairs of the energy: the ni x nj pairs of a cell with another one (or
// with itself, `same`: each pair once) in square tiles.  Tiles of a cell pair,
// and rows and columns of tile k (the cell itself: tiles on and below the
// diagonal).
#define MC_NEAR_TILE 128
__host__ __device__ __forceinline__ long long near_tiles(int ni, int nj, bool same, int tile = MC_NEAR_TILE) {
  const long long a = (ni + tile - 1) / tile, b = (nj + tile - 1) / tile;
  return same ? a * (a + 1) / 2 : a * b;
}
__host__ __device__ __forceinline__ void near_tile(long long k, int nj, bool same, int* ti, int* tj,
                                                  int tile = MC_NEAR_TILE) {
  if (same) {
    long long i = (long long)((sqrt(8.0 * (double)k + 1.0) - 1.0) * 0.5);
    while (i * (i + 1) / 2 > k) i--;
    while ((i + 1) * (i + 2) / 2 <= k) i++;
    *ti = (int)i;
    *tj = (int)(k - i * (i + 1) / 2);
  } else {
    const long long b = (nj + tile - 1) / tile;
    *ti = (int)(k / b);
    *tj = (int)(k % b);
  }
}
