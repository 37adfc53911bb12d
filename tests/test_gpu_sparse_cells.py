"""Energies of systems with few charges and many cells: against the oracle in
both methods, whichever way (cell by cell or particle by particle) the number
of charges asks for, and the time of a fresh energy.

A fresh energy of a thousand charges on 7 levels is 0.1 ms of work for a warp per
charge; cell by cell it took 3.5 ms.  The bound, 1.5 ms, leaves room for a slow
host.
"""
import time

import numpy as np
import pytest

import oracle as O
from paper_2006_16622_gb300 import mcfmm
from paper_2006_16622_gb300.workloads import uniform_system

pytestmark = pytest.mark.gpu

PBC, FREE = mcfmm.BC_PBC, mcfmm.BC_FREE


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    mcfmm.load()


# 64 and 512 cells; 48 and 384 charges are 3/4 of one a cell
@pytest.mark.parametrize("n,L", [(2, 3), (46, 3), (48, 3), (50, 3), (10, 4), (382, 4), (384, 4), (512, 4), (40, 5)])
@pytest.mark.parametrize("bc", [PBC, FREE])
def test_energies_of_few_charges(n, L, bc):
    a, p = 7.0, 6
    pos, q = uniform_system(n, a, seed=n)
    o = O.System(pos, q, a, L, p, bc=bc)
    o.setup()
    tol = 1e-10 * max(1.0, abs(o.energy()))
    g = mcfmm.Context(pos, q, a, L, p, bc=bc)
    g.setup(mcfmm.SETUP_P2L)
    assert abs(g.energy() - o.energy()) <= tol and abs(g.energy_fresh() - o.energy()) <= tol
    # the same expansions contracted the other way round
    g.setup(mcfmm.SETUP_MULTIPOLE)
    assert abs(g.energy() - o.energy()) <= tol and abs(g.energy_fresh() - o.energy()) <= tol
    g.close()


def test_fresh_energy_of_few_charges_is_quick():
    pos, q = uniform_system(1000, 20.0, seed=1)
    g = mcfmm.Context(pos, q, 20.0, 7, 8)
    g.setup(mcfmm.SETUP_P2L)
    t = []
    for _ in range(9):
        t0 = time.perf_counter()
        g.energy_fresh()
        t.append(time.perf_counter() - t0)
    g.close()
    assert np.median(t) < 1.5e-3, t


# half of the charges in one cell, around the line between the two ways (2000 at
# L = 3, 4000 at L = 4)
@pytest.mark.parametrize("n,L", [(300, 3), (1998, 3), (2000, 3), (3998, 4), (4000, 4)])
def test_energies_beside_a_dense_cell(n, L):
    a, p = 9.0, 4
    pos, q = uniform_system(n, a, seed=L)
    pos[:n // 2] = (0.01 + 0.98 * np.random.default_rng(n).uniform(size=(n // 2, 3))) * (a / (1 << (L - 1)))
    o = O.System(pos, q, a, L, p, bc=FREE)
    o.setup()
    tol = 1e-10 * max(1.0, abs(o.energy()))
    g = mcfmm.Context(pos, q, a, L, p, bc=FREE)
    g.setup(mcfmm.SETUP_P2L)
    assert abs(g.energy() - o.energy()) <= tol and abs(g.energy_fresh() - o.energy()) <= tol
    g.close()


def test_fresh_energy_of_a_small_dense_system_is_quick():
    """2000 of 4000 charges in one cell: 0.29 ms for a warp per charge, 0.98 ms cell
    by cell in tiles of 128 x 128 pairs"""
    n, a, L = 4000, 30.0, 5
    pos, q = uniform_system(n, a, seed=4)
    pos[:n // 2] = (0.01 + 0.98 * np.random.default_rng(3).uniform(size=(n // 2, 3))) * (a / (1 << (L - 1)))
    g = mcfmm.Context(pos, q, a, L, 8, bc=FREE)
    g.setup(mcfmm.SETUP_P2L)
    t = []
    for _ in range(9):
        t0 = time.perf_counter()
        g.energy_fresh()
        t.append(time.perf_counter() - t0)
    g.close()
    assert np.median(t) < 0.6e-3, t
