"""The fixed-point harmonic sums (csrc/mc_fix.cuh) on the CPU.

The header compiles for the host; the harness runs exactly what one lane and
one thread of the kernel run (charge set-up, powers of e^{i phi} and of
rho sin t, the recurrence of every column, the multiply-accumulate) and
compares every scaled coefficient with the two-term recurrences in
long double, over displacements of the whole range: near the axis, on the
faces and corners of the nearest listed cells, at the furthest corner.

Bound: a term's error in units of the largest value its coefficient can have
(R0^-(n+1) or R0^n in the paper's normalisation).  Products are rounded at
2^-58; the scale factors are doubles (2^-53 of the value); the recurrence
loses at most the ratio of a harmonic's largest value to its size at the
start of its column (below 2^8 for p <= 15) times 2^-59.  So rms < 2^-54 and
every term < 2^-49.
"""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2006_16622_gb300", "csrc")

HARNESS = r"""
#define __host__
#define __device__
#define __forceinline__ inline
#include "mc_fix.cuh"
#include <cstdio>
#include <cstdlib>
#include <vector>
typedef long double Q;

static void reference(int p, bool irr, Q x, Q y, Q z, std::vector<Q>& re, std::vector<Q>& im) {
  Q r2 = x * x + y * y + z * z, u = x, v = y, w = z, s = r2, start = 1;
  if (irr) {
    const Q g = sqrtl(r2);
    u = x / r2; v = y / r2; w = z / r2; s = 1 / r2; start = 1 / g;
  }
  re.assign((p + 1) * (p + 1), 0);
  im.assign((p + 1) * (p + 1), 0);
  Q dr = start, di = 0;
  for (int m = 0; m <= p; m++) {
    if (m) {
      const Q f = irr ? (Q)(2 * m - 1) : 1 / (Q)(2 * m), nr = f * (dr * u - di * v), ni = f * (dr * v + di * u);
      dr = nr;
      di = ni;
    }
    Q a0r = 0, a0i = 0, a1r = dr, a1i = di;
    for (int n = m; n <= p; n++) {
      if (n > m) {
        Q A, B;
        if (irr) { A = 2 * n - 1; B = (Q)(n + m - 1) * (n - m - 1); }
        else { const Q den = (Q)(n + m) * (n - m); A = (2 * n - 1) / den; B = 1 / den; }
        const Q cr = A * w * a1r - B * s * a0r, ci = A * w * a1i - B * s * a0i;
        a0r = a1r; a0i = a1i; a1r = cr; a1i = ci;
      }
      re[n * n + m] = a1r;
      im[n * n + m] = a1i;
    }
  }
}
static double rnd() { return rand() / (RAND_MAX + 1.0); }

int main(int argc, char** argv) {
  const int p = atoi(argv[1]);
  const bool irr = atoi(argv[2]);
  srand(11 + p);
  const double w = 1.7;
  FixTab T;
  fix_tab_build(&T, p, irr, irr ? kFixR0 * w : w);
  const FixShares sh = fix_shares(p);
  // every coefficient once, within the steps of one warp
  std::vector<int> seen((p + 1) * (p + 1), 0);
  for (int k = 0; k < MC_FIX_WARPS; k++)
    for (int t = 0; t < MC_FIX_STEPS; t++)
      if (T.index[k][t] >= 0) {
        if (t >= sh.steps || T.step[k][t].wh >= 0x80000000u) return 2;
        seen[T.index[k][t]]++;
      }
  for (int n = 0; n <= p; n++)
    for (int m = 0; m <= n; m++)
      if (seen[n * n + (m ? 2 * m - 1 : 0)] != 1) return 3;
  double worst = 0, sq = 0;
  long cnt = 0;
  std::vector<Q> re, im;
  for (int k = 0; k < 2000; k++) {
    int64_t D[3];
    Q X[3];
    double v[3];
    do {
      for (int d = 0; d < 3; d++) v[d] = irr ? rnd() * 7 - 3.5 : rnd() - 0.5;
      if (k % 4 == 1) { v[0] *= 1e-5; v[1] *= k % 8 == 1 ? 0.0 : 1e-9; }  // near the axis
      if (k % 4 == 2) {                                                    // faces and corners
        for (int d = 0; d < 3; d++) v[d] = (irr ? (rand() % 2 ? 1.5 : 3.5) : 0.5) * (rand() % 2 ? 1 : -1);
        if (rand() % 2) v[rand() % 3] *= rnd();
      }
    } while (irr && fabs(v[0]) < 1.5 && fabs(v[1]) < 1.5 && fabs(v[2]) < 1.5);
    for (int d = 0; d < 3; d++) {
      D[d] = (int64_t)(v[d] / (irr ? 4.0 : 1.0) * 4611686018427387904.0);
      X[d] = (Q)D[d] / 4611686018427387904.0L * (irr ? 4 : 1) * w;
    }
    const double q = k % 2 ? 1.0 : -0.7;
    const FixCharge c = irr ? fix_irregular(D[0], D[1], D[2], fx_charge(q, 1023))
                            : fix_regular(D[0], D[1], D[2], fx_charge(q, 1023));
    reference(p, irr, X[0], X[1], X[2], re, im);
    const Fx ex = fx_split(c.ex), ey = fx_split(c.ey), en = fx_split(-c.ey), st = fx_split(c.st);
    int64_t y = c.x0, xr = (int64_t)1 << 62, xi = 0;
    for (int m = 0; m <= p; m++) {
      const Fx pr = fx_split(xr >> MC_FIX_PHASE), pi = fx_split(xi >> MC_FIX_PHASE), zp = fx_split(c.zeta), zn = fx_split(-c.zeta);
      Fx q1 = fx_split(y), q2 = {0, 0};
      for (int n = m; n <= p; n++) {
        const int i = n - m, t = sh.first[m] + i, wi = sh.warp[m];
        if (i) {
          const FixStep& s = T.step[wi][t];
          const Fx qq = fix_next((i & 1) ? zp : zn, (uint32_t)(c.kap >> 32), (uint32_t)c.kap, q1, q2, s.wh, s.wl, s.sh);
          q2 = q1;
          q1 = qq;
        }
        const long double sc = (long double)T.scale[wi][t] / 32.0L;
        long double f = 1, f2 = 1;
        for (int j = 1; j <= n - m; j++) f *= j;
        for (int j = 1; j <= n + m; j++) f2 *= j;
        const long double R = irr ? kFixR0 * w : w;
        const long double unit = irr ? sqrtl(f * f2) * powl(R, -(n + 1)) : powl(R, n) / sqrtl(f * f2);
        const double er = (double)(((Q)fix_mac(pr, q1, 0) * sc - (Q)q * re[n * n + m]) / unit);
        const double ei = (double)(((Q)fix_mac(pi, q1, 0) * sc - (Q)q * im[n * n + m]) / unit);
        worst = fmax(worst, fmax(fabs(er), fabs(ei)));
        sq += er * er + ei * ei;
        cnt += 2;
      }
      y = fx_mul62(fx_split(y), st);
      fx_turn(fx_split(xr), fx_split(xi), ex, ey, en, &xr, &xi);
    }
  }
  printf("%.17g %.17g\n", sqrt(sq / cnt), worst);
  return 0;
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("fix")
    src, exe = d / "h.cpp", d / "h"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-O2", "-std=gnu++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    return str(exe)


@pytest.mark.parametrize("irregular", [1, 0])
@pytest.mark.parametrize("p", [0, 1, 2, 7, 8, 11, 12, 15])
def test_terms_against_quadruple_precision(harness, p, irregular):
    out = subprocess.run([harness, str(p), str(irregular)], capture_output=True, text=True)
    assert out.returncode == 0, out
    rms, worst = (float(x) for x in out.stdout.split())
    assert rms < 2.0 ** -54 and worst < 2.0 ** -49
