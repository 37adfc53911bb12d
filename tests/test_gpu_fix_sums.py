"""The setup's fixed-point harmonic sums on the GPU where they can go wrong:
every kernel instantiation (p = 0..15), levels with one chunk and with many,
fewer charges than a staged batch, empty cells, free space, and the charges
that go to the FP64 gather instead (sizes further apart than 2^6; rows that do
not lie in their cell).

Tolerance 1e-12 of the level's largest coefficient, that of the other parity
tests: a fixed-point term is within 2^-49 of the largest coefficient a charge
can have (the bound of the CPU test of the same arithmetic), and rounding
errors of the ~190 x 20 charges of a list add up to less than 70 times that.
"""
import numpy as np
import pytest

import oracle as O
from paper_2006_16622_gb300 import mcfmm
from paper_2006_16622_gb300.workloads import uniform_system

pytestmark = pytest.mark.gpu

TOL = 1e-12


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    mcfmm.load()


def _same(got, ref, what):
    assert np.max(np.abs(got - ref)) <= TOL * max(np.max(np.abs(ref)), 1e-300), what


def _check(pos, q, a, L, p, bc=mcfmm.BC_PBC):
    g = mcfmm.Context(pos, q, a, L, p, bc=bc)
    g.setup()
    o = O.System(pos, q, a, L, p, bc=bc)
    o.setup()
    for lev in range(2, L + 1):
        _same(g.local(lev), o.local(lev), lev)
    assert abs(g.energy() - o.energy()) <= 1e-10 * max(1.0, abs(o.energy()))
    g.close()


@pytest.mark.parametrize("p", range(16))
def test_every_order(p):
    pos, q = uniform_system(210, 7.3, seed=p)
    _check(pos, q, 7.3, 3, p)


@pytest.mark.parametrize("n,L,p,bc", [(2, 2, 5, mcfmm.BC_PBC), (6, 4, 12, mcfmm.BC_PBC), (34, 3, 9, mcfmm.BC_FREE),
                                      (1500, 2, 11, mcfmm.BC_PBC), (900, 5, 8, mcfmm.BC_FREE), (2600, 4, 13, mcfmm.BC_PBC)])
def test_few_and_many_charges(n, L, p, bc):
    a = 3.7e-3  # a box far from unit size
    pos, q = uniform_system(n, a, seed=n)
    g = mcfmm.Context(pos, q, a, L, p, bc=bc)
    g.setup()
    o = O.System(pos, q, a, L, p, bc=bc)
    o.setup()
    for lev in range(2, L + 1):
        _same(g.local(lev), o.local(lev), lev)


def _paired(q, factor):
    """charges scaled in pairs (one +, one -), so that they stay neutral"""
    q = q.copy()
    plus, minus = np.nonzero(q > 0)[0], np.nonzero(q < 0)[0]
    q[plus] *= factor
    q[minus] *= factor
    return q


@pytest.mark.parametrize("span", [4.0, 60.0, 1e5])
def test_uneven_charges(span):
    n, a, L, p = 400, 9.0, 3, 10
    pos, q = uniform_system(n, a, seed=5)
    f = np.exp(np.random.default_rng(1).uniform(0.0, np.log(span), n // 2))
    _check(pos, _paired(q, f), a, L, p)


def _level(part, start, n, a, L, lev, p):
    import torch
    out = torch.empty((8 ** (lev - 1), (p + 1) ** 2), dtype=torch.float64, device="cuda")
    d_part, d_start = torch.tensor(part, device="cuda"), torch.tensor(start, device="cuda")
    rc = mcfmm.p2l_level_noalloc(d_part.data_ptr(), d_start.data_ptr(), n, a, L, lev, p, mcfmm.BC_PBC, out.data_ptr(),
                                 torch.cuda.current_stream().cuda_stream)
    assert rc == 0
    return out.cpu().numpy()


def _rows(pos, q, a, L):
    nL = 1 << (L - 1)
    c = np.minimum(np.floor(pos * (nL / a)).astype(np.int64), nL - 1)
    cell = (c[:, 0] * nL + c[:, 1]) * nL + c[:, 2]
    order = np.argsort(cell, kind="stable")
    part = np.ascontiguousarray(np.concatenate([pos[order], q[order, None]], axis=1))
    return part, np.searchsorted(cell[order], np.arange(nL ** 3 + 1)).astype(np.int32)


@pytest.mark.parametrize("factor", [1.0, 1e4])
def test_noalloc_even_and_uneven(factor):
    n, a, L, p = 700, 9.0, 3, 9
    pos, q = uniform_system(n, a, seed=8)
    q = _paired(q, np.where(np.arange(n // 2) % 7 == 0, factor, 1.0))
    part, start = _rows(pos, q, a, L)
    o = O.System(pos, q, a, L, p)
    o.setup()
    for lev in (2, 3):
        _same(_level(part, start, n, a, L, lev, p), o.local(lev), lev)


def test_noalloc_row_outside_its_cell():
    """such rows are summed as they are, as by the FP64 gather (forced here by
    a charge of 1e-12, whose own part is below the tolerance)"""
    n, a, L, p = 700, 9.0, 3, 9
    pos, q = uniform_system(n, a, seed=8)
    pos[3] = [a * 1.01, 0.3 * a, 0.4 * a]
    part, start = _rows(pos, q, a, L)
    forced = part.copy()
    forced[10, 3] = 1e-12
    part[10, 3] = 0.0
    for lev in (2, 3):
        _same(_level(part, start, n, a, L, lev, p), _level(forced, start, n, a, L, lev, p), lev)
