"""Tiles of the energy's near pairs (csrc/mc_fix.cuh near_tiles, near_tile) on
the CPU: every pair of two cells, or of a cell with itself, lies in exactly
one tile, for counts around the tile's 128.
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
#include <algorithm>
#include <cstdio>
#include <vector>
int main() {
  const int n[] = {0, 1, 2, 127, 128, 129, 255, 256, 257, 400, 1000};
  for (int ni : n)
    for (int nj : n)
      for (int same = 0; same < 2; same++) {
        if (same && ni != nj) continue;
        std::vector<int> seen((size_t)ni * nj, 0);
        for (long long k = 0; k < near_tiles(ni, nj, same); k++) {
          int ti, tj;
          near_tile(k, nj, same, &ti, &tj);
          for (int i = ti * MC_NEAR_TILE; i < std::min(ni, (ti + 1) * MC_NEAR_TILE); i++)
            for (int j = tj * MC_NEAR_TILE; j < std::min(nj, (tj + 1) * MC_NEAR_TILE); j++)
              if (!same || j < i) seen[(size_t)i * nj + j]++;
        }
        for (int i = 0; i < ni; i++)
          for (int j = 0; j < nj; j++)
            if (seen[(size_t)i * nj + j] != (!same || j < i)) return 1;
      }
  // far along a large diagonal
  for (long long i : {1ll, 4096ll, 8000000ll})
    for (long long k : {i * (i + 1) / 2 - 1, i * (i + 1) / 2, i * (i + 1) / 2 + i}) {
      int ti, tj;
      near_tile(k, 1 << 30, true, &ti, &tj);
      if ((long long)ti * (ti + 1) / 2 + tj != k || tj < 0 || tj > ti) return 2;
    }
  return 0;
}
"""


def test_every_pair_in_one_tile(tmp_path):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    src, exe = tmp_path / "h.cpp", tmp_path / "h"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-O2", "-std=gnu++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0
