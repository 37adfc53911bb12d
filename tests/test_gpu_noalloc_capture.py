"""The allocation-free level call under stream capture: the first call of the
process (another order, before the capture, as the header asks for) and then a
captured one whose order's kernels have not run yet; the replayed graph works
on what its buffers hold then.  In a process of its own, so that no other test
has loaded those kernels.
"""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CODE = r"""
import numpy as np, torch
from paper_2006_16622_gb300 import mcfmm
from paper_2006_16622_gb300.workloads import uniform_system

def rows(pos, q, a, L):
    nL = 1 << (L - 1)
    c = np.minimum(np.floor(pos * (nL / a)).astype(np.int64), nL - 1)
    cell = (c[:, 0] * nL + c[:, 1]) * nL + c[:, 2]
    order = np.argsort(cell, kind="stable")
    return (torch.tensor(np.concatenate([pos[order], q[order, None]], axis=1), device="cuda"),
            torch.tensor(np.searchsorted(cell[order], np.arange(nL ** 3 + 1)).astype(np.int32), device="cuda"))

def call(part, start, p, out):
    rc = mcfmm.p2l_level_noalloc(part.data_ptr(), start.data_ptr(), len(part), a, L, 3, p, mcfmm.BC_PBC,
                                 out.data_ptr(), torch.cuda.current_stream().cuda_stream)
    assert rc == 0, rc

a, L = 9.0, 3
first, second = [rows(*uniform_system(500, a, seed=s), a, L) for s in (1, 2)]
call(*first, 3, torch.empty((64, 16), dtype=torch.float64, device="cuda"))
torch.cuda.synchronize()
for p in (5, 11):
    part, start = first[0].clone(), first[1].clone()
    out = torch.zeros((64, (p + 1) ** 2), dtype=torch.float64, device="cuda")
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        call(part, start, p, out)
    for src in (first, second):
        part.copy_(src[0])
        start.copy_(src[1])
        out.zero_()
        g.replay()
        torch.cuda.synchronize()
        ref = torch.zeros_like(out)
        call(*src, p, ref)
        torch.cuda.synchronize()
        assert torch.equal(out, ref) and float(ref.abs().max()) > 0.0, p
print("captured")
"""


def test_capture_of_an_order_not_used_before():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CODE], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "captured" in r.stdout, r.stdout + r.stderr
