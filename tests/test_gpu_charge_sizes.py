"""Charges at the ends of the exponent range: subnormal ones, and ones whose
next power of two is no double.  Everything linear in the charges is the same
as for unit charges, times a power of two.

1e-12 of the level's largest coefficient, as in the other parity tests.
"""
import numpy as np
import pytest

from paper_2006_16622_gb300 import mcfmm
from paper_2006_16622_gb300.workloads import uniform_system

pytestmark = pytest.mark.gpu

L, P = 3, 4


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    mcfmm.load()


def _level(pos, q, a, lev):
    import torch
    nL = 1 << (L - 1)
    c = np.minimum(np.floor(pos * (nL / a)).astype(np.int64), nL - 1)
    cell = (c[:, 0] * nL + c[:, 1]) * nL + c[:, 2]
    order = np.argsort(cell, kind="stable")
    part = torch.tensor(np.concatenate([pos[order], q[order, None]], axis=1), device="cuda")
    start = torch.tensor(np.searchsorted(cell[order], np.arange(nL ** 3 + 1)).astype(np.int32), device="cuda")
    out = torch.empty((8 ** (lev - 1), (P + 1) ** 2), dtype=torch.float64, device="cuda")
    rc = mcfmm.p2l_level_noalloc(part.data_ptr(), start.data_ptr(), len(q), a, L, lev, P, mcfmm.BC_PBC, out.data_ptr(),
                                 torch.cuda.current_stream().cuda_stream)
    assert rc == 0
    return out.cpu().numpy()


def _scaled(x, e):
    """x 2^e with every step exact"""
    return np.ldexp(np.ldexp(x, e // 2), e - e // 2)


# box sides: every product of the sums stays a normal number
@pytest.mark.parametrize("e,a", [(-1040, 1e-6), (-1060, 1e-15), (1023, 2.0 ** 100)])
def test_level_without_allocation(e, a):
    pos, q = uniform_system(300, a, seed=4)
    q = q / np.abs(q)
    for lev in (2, 3):
        ref = _level(pos, q, a, lev)
        got = _scaled(_level(pos, _scaled(q, e), a, lev), -e)
        assert np.max(np.abs(got - ref)) <= 1e-12 * np.max(np.abs(ref)), lev


@pytest.mark.parametrize("e,a", [(-1040, 1e-6), (-1060, 1e-15)])
@pytest.mark.parametrize("mode", [mcfmm.SETUP_P2L, mcfmm.SETUP_MULTIPOLE])
def test_setup(e, a, mode):
    pos, q = uniform_system(300, a, seed=4)
    q = q / np.abs(q)
    got = []
    for x in (q, _scaled(q, e)):
        c = mcfmm.Context(pos, x, a, L, P)
        c.setup(mode)
        # (multipoles: the monopoles, small integers times the charge, stay exact)
        got.append([c.multipole(l)[:, :1] if mode == mcfmm.SETUP_MULTIPOLE else c.local(l) for l in (2, 3)])
        c.close()
    for ref, x in zip(*got):
        assert np.max(np.abs(_scaled(x, -e) - ref)) <= 1e-12 * np.max(np.abs(ref))
