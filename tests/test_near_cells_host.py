"""Coordinates of the energy's near pairs (csrc/mc_fix.cuh fx_cells) on the
CPU: units of 2^-60 finest cells modulo 2^64, rounded down by less than two,
against exact rational arithmetic, for every number of levels and coordinates
from the lower face to the upper one.
"""
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
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
int main(int argc, char** argv) {
  const double a = strtod(argv[1], nullptr);
  const int L = atoi(argv[2]);
  uint64_t u;
  __builtin_memcpy(&u, &a, 8);
  const uint64_t m = (u & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull;
  const unsigned __int128 top = (unsigned __int128)1 << 115;
  const uint64_t r1 = (uint64_t)(top / m), r0 = (uint64_t)((top % m << 64) / m);
  for (int i = 3; i < argc; i++)
    printf("%llu\n", (unsigned long long)fx_cells(strtod(argv[i], nullptr), r1, r0, (int)((u >> 52) & 0x7ff), L));
  return 0;
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("cells")
    src, exe = d / "h.cpp", d / "h"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-O2", "-std=gnu++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    return str(exe)


@pytest.mark.parametrize("L", range(2, 9))
@pytest.mark.parametrize("a", [7.99999999, 8.0, 46.4, 1.0, 3.7e-3])
def test_coordinate(harness, L, a):
    xs = [0.0, np.nextafter(a, 0.0)] + [f * a for f in (1e-300, 1e-19, 1e-17, 1e-9, 1e-3)]
    xs += list(np.random.default_rng(L).uniform(0.0, a, 100)) + list(a * 2.0 ** np.random.default_rng(L).uniform(-12, 0, 100))
    out = subprocess.run([harness, float(a).hex(), str(L)] + [float(x).hex() for x in xs], capture_output=True, text=True, check=True)
    for x, got in zip(xs, out.stdout.split()):
        exact = Fraction(float(x)) / Fraction(a) * 2 ** (59 + L)
        below = (exact - int(got)) % 2 ** 64
        assert below < 2 or below > 2 ** 64 - Fraction(1, 1000), (x / a, float(below))
