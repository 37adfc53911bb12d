"""The allocation-free level call takes its rows from the cell offsets alone:
the row count it is given, which the header calls informational, changes not a
bit of the result (nor the split of the work that decides the bits).
"""
import numpy as np
import pytest

from paper_2006_16622_gb300 import mcfmm
from paper_2006_16622_gb300.workloads import uniform_system

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    mcfmm.load()


@pytest.mark.parametrize("n,L", [(40, 4), (1000, 3), (20000, 2), (20000, 4)])
def test_count_of_rows_is_informational(n, L):
    import torch
    a, p = 9.0, 6
    nL = 1 << (L - 1)
    pos, q = uniform_system(n, a, seed=L)
    c = np.minimum(np.floor(pos * (nL / a)).astype(np.int64), nL - 1)
    cell = (c[:, 0] * nL + c[:, 1]) * nL + c[:, 2]
    order = np.argsort(cell, kind="stable")
    part = torch.tensor(np.concatenate([pos[order], q[order, None]], axis=1), device="cuda")
    start = torch.tensor(np.searchsorted(cell[order], np.arange(nL ** 3 + 1)).astype(np.int32), device="cuda")
    for lev in range(2, L + 1):
        out = []
        for rows in (n, 0, 1000 * n):
            o = torch.empty((8 ** (lev - 1), (p + 1) ** 2), dtype=torch.float64, device="cuda")
            assert mcfmm.p2l_level_noalloc(part.data_ptr(), start.data_ptr(), rows, a, L, lev, p, mcfmm.BC_PBC, o.data_ptr(),
                                           torch.cuda.current_stream().cuda_stream) == 0
            out.append(o.cpu().numpy())
        assert np.array_equal(out[0], out[1]) and np.array_equal(out[0], out[2]), lev
