"""Box coordinates of the fixed-point sums (csrc/mc_fix.cuh fx_coord) on the
CPU: x / a in units of 2^-62 against exact rational arithmetic, for box sides
on both sides of a power of two and x from 0 to 2^-14 beyond the upper face.

Bound: the reciprocal is rounded at 2^-63 of itself, the product and the final
shift round down, and a row beyond the face with the next exponent loses one
more bit: within 4 units.
"""
import os
import shutil
import subprocess
from fractions import Fraction

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
  uint64_t u;
  __builtin_memcpy(&u, &a, 8);
  const uint64_t m = (u & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull;
  const uint64_t rcp = (uint64_t)((((unsigned __int128)1 << 115) + m / 2) / m);
  for (int i = 2; i < argc; i++)
    printf("%lld\n", (long long)fx_coord(strtod(argv[i], nullptr), rcp, (int)((u >> 52) & 0x7ff)));
  return 0;
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("coord")
    src, exe = d / "h.cpp", d / "h"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-O2", "-std=gnu++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    return str(exe)


@pytest.mark.parametrize("a", [7.99999999, 8.0, 8.00000001, 6.0, 1.9999999999999998, 1.0, 3.7e-3, 0.99999 * 2.0 ** -40])
def test_coordinate(harness, a):
    xs = [f * a for f in (0.0, 1e-17, 1e-3, 0.3, 0.5, 0.9999, 1.0, 1.0 + 2.0 ** -30, 1.0 + 2.0 ** -20, 1.0 + 2.0 ** -14)]
    out = subprocess.run([harness, a.hex()] + [x.hex() for x in xs], capture_output=True, text=True, check=True)
    for x, got in zip(xs, out.stdout.split()):
        assert abs(int(got) - Fraction(x) / Fraction(a) * 2 ** 62) <= 4, (x / a, got)
