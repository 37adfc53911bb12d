"""The allocation-free level call with rows a little beyond the upper face of
the box (its cell rule clamps them into the last cell) in a box whose side is
just below a power of two, so that such a coordinate has a larger exponent
than the side.  They are summed where they are.

Against the FP64 gather (forced by one charge of 1e-12, whose own part is below
the tolerance), 1e-12 of the level's largest coefficient as in the other parity
tests.
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


def _level(part, start, a, L, lev, p):
    import torch
    out = torch.empty((8 ** (lev - 1), (p + 1) ** 2), dtype=torch.float64, device="cuda")
    d_part, d_start = torch.tensor(part, device="cuda"), torch.tensor(start, device="cuda")
    rc = mcfmm.p2l_level_noalloc(d_part.data_ptr(), d_start.data_ptr(), len(part), a, L, lev, p, mcfmm.BC_PBC, out.data_ptr(),
                                 torch.cuda.current_stream().cuda_stream)
    assert rc == 0
    return out.cpu().numpy()


@pytest.mark.parametrize("a", [7.99999999, 8.0, 6.0, 3.9999999999])
@pytest.mark.parametrize("beyond", [1e-9, 0.9 / 16384.0])  # in finest cells
def test_row_beyond_the_upper_face(a, beyond):
    L, p = 3, 9
    nL = 1 << (L - 1)
    pos, q = uniform_system(400, a, seed=8)
    pos[3, 0] = pos[7, 1] = pos[11, 2] = a + beyond * a / nL
    c = np.minimum(np.floor(pos * (nL / a)).astype(np.int64), nL - 1)
    cell = (c[:, 0] * nL + c[:, 1]) * nL + c[:, 2]
    order = np.argsort(cell, kind="stable")
    part = np.ascontiguousarray(np.concatenate([pos[order], q[order, None]], axis=1))
    start = np.searchsorted(cell[order], np.arange(nL ** 3 + 1)).astype(np.int32)
    part[10, 3] = 0.0
    forced = part.copy()
    forced[10, 3] = 1e-12
    for lev in (2, 3):
        got, ref = _level(part, start, a, L, lev, p), _level(forced, start, a, L, lev, p)
        assert np.max(np.abs(got - ref)) <= 1e-12 * np.max(np.abs(ref)), lev
