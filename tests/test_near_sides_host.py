"""The barrier-free FP64 chain's near items (csrc/mc_geom.cuh near_part_sides)
on the CPU: 54 P items, one side of one of the 27 near cells each, sum every
slot of a cell exactly once for each side, for every split P = 1..4 and cell
occupancy (slot 32 part + lane, stepping by 32 P, 32 lanes).  No GPU.
"""
import shutil
import subprocess

import pytest

from test_near_split_host import HARNESS, HEADER, _coverage


@pytest.mark.parametrize("P", [1, 2, 3, 4])
def test_every_slot_once(tmp_path, P):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    src, exe = tmp_path / "h.cpp", tmp_path / "h"
    src.write_text(HARNESS.replace("HEADER", HEADER).replace("near_part(k0, same, nparts, nsame)",
                                                            "near_part_sides(k0, nparts)"))
    subprocess.run([gxx, "-std=c++17", "-O1", "-o", str(exe), str(src)], check=True)
    out = subprocess.run([str(exe), str(54 * P), "0", str(P), "0"], check=True, capture_output=True, text=True).stdout
    items = [tuple(int(v) for v in line.split()) for line in out.splitlines()]
    assert len(items) == 54 * P
    for cnt in (0, 1, 31, 32, 33, 63, 64, 65, 100, 190, 255, 256, 384):
        cov = _coverage(items, cnt)
        for k in range(27):
            for side in (0, 1):
                assert sorted(cov.get((k, side), [])) == list(range(cnt)), (k, side, cnt)
