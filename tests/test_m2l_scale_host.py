"""Powers of two of the fixed-point multipole-to-local translations
(csrc/mc_m2l_scale.cuh) on the CPU: with them no entry of a matrix exceeds 1
and no row sums to more than 126 over the offsets of a group and all columns,
which is what 59-bit entries, 57-bit multipoles and 64-bit sums leave room for.
The order 15 covers the lower ones (their rows are parts of its rows).
"""
import math
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2006_16622_gb300", "csrc")
P = 15

HARNESS = r"""
#define __host__
#define __device__
#define __constant__
#define __forceinline__ inline
#include "mc_m2l_scale.cuh"
#include <cstdio>
int main() {
  for (int n = 0; n < 16; n++) std::printf("%d ", kM2LColScale[n]);
  for (int g = 0; g < MC_M2L_GROUPS; g++)
    for (int j = 0; j < 16; j++) std::printf("%d ", kM2LRowScale[g][j]);
  for (int o = 0; o < 64; o++) std::printf("%d ", m2l_group(o));
}
"""


def _irregular(o, lmax):
    """I_l^m(o) = (l - m)! P_l^m e^{i m phi} / r^(l+1), m >= 0"""
    x, y, z = (float(v) for v in o)
    i2 = 1.0 / (x * x + y * y + z * z)
    out = np.zeros((lmax + 1, lmax + 1), complex)
    c = math.sqrt(i2) + 0j
    for m in range(lmax + 1):
        if m:
            c *= (2 * m - 1) * i2 * (x + 1j * y)
        b, g = 0j, c
        for n in range(m, lmax + 1):
            if n > m:
                b, g = g, i2 * ((2 * n - 1) * z * g - ((n - 1) ** 2 - m * m) * b)
            out[n, m] = g
    return out


def _matrix(o):
    """|T| of the real layout, paper normalisation, unit cells"""
    I = _irregular(o, 2 * P)
    s = [[math.sqrt(math.factorial(n - m) * math.factorial(n + m)) for m in range(n + 1)] for n in range(P + 1)]
    get = lambda l, m: I[l, m] if m >= 0 else (-1) ** m * np.conj(I[l, -m])
    T = np.zeros(((P + 1) ** 2,) * 2)
    for n in range(P + 1):
        for m in range(n + 1):
            for j in range(P + 1):
                for k in range(j + 1):
                    r, c = j * j + (2 * k - 1 if k else 0), n * n + (2 * m - 1 if m else 0)
                    a, b = get(j + n, k + m), (-1) ** m * get(j + n, k - m) if m else 0j
                    f = 1.0 / (s[n][m] * s[j][k])
                    T[r, c] = abs((a + b).real) * f
                    if m:
                        T[r, c + 1] = abs((a - b).imag) * f
                    if k:
                        T[r + 1, c] = abs((a + b).imag) * f
                        if m:
                            T[r + 1, c + 1] = abs((a - b).real) * f
    return T


def test_sums_fit(tmp_path):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    src, exe = tmp_path / "h.cpp", tmp_path / "h"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-O2", "-std=gnu++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    v = np.array(subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split(), dtype=int)
    groups = (len(v) - 16 - 64) // 16
    col, row, grp = v[:16], v[16:16 + 16 * groups].reshape(groups, 16), v[16 + 16 * groups:]
    deg = np.repeat(np.arange(16), 2 * np.arange(16) + 1)
    sums, peak, seen = np.zeros((groups, 256)), np.zeros(groups), set()
    for code in range(64):
        o = (code & 3, (code >> 2) & 3, code >> 4)
        if max(o) < 2:
            continue
        g = grp[code]
        seen.add(g)
        T = np.ldexp(_matrix(o), row[g][deg][:, None] - col[deg][None, :])
        # signs that a list of a cell holds: both of 1 and 2, one of 3
        members = math.prod(2 if c in (1, 2) else 1 for c in o)
        sums[g] += members * T.sum(1)
        peak[g] = max(peak[g], T.max())
    assert seen == set(range(groups))
    assert sums.max() <= 126.0 and peak.max() <= 1.0
    # and no power is smaller than it has to be
    assert np.all((sums.reshape(groups, -1).max(1) > 31.0) | (peak > 0.25))
