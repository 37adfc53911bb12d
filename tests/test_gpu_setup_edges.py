"""The setups on the GPU at the edges of their kernels: lowest and highest
orders of the fast setup's translations and of the multipoles' way up, the
smallest trees, free space, charges too uneven for the fixed-point sums, and
the energy's near pairs for particle counts around the lanes of a warp.

Tolerances of the other parity tests: arrays 1e-12 of the largest coefficient
of their level, energies 1e-10.
"""
import numpy as np
import pytest

import oracle as O
from paper_2006_16622_gb300 import mcfmm
from paper_2006_16622_gb300.workloads import uniform_system

pytestmark = pytest.mark.gpu

ARR_TOL, E_TOL = 1e-12, 1e-10
PBC, FREE = mcfmm.BC_PBC, mcfmm.BC_FREE


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    mcfmm.load()


def _same(got, ref, what):
    assert np.max(np.abs(got - ref)) <= ARR_TOL * np.max(np.abs(ref)), what


def _energies(g, o):
    assert abs(g.energy() - o.energy()) <= E_TOL * max(1.0, abs(o.energy()))
    assert abs(g.energy_fresh() - o.energy()) <= E_TOL * max(1.0, abs(o.energy()))


def _uneven(q):
    """charges over 1e5, scaled in neutral pairs"""
    f = np.exp(np.random.default_rng(1).uniform(0.0, np.log(1e5), len(q) // 2))
    q = q.copy()
    q[np.nonzero(q > 0)[0]] *= f
    q[np.nonzero(q < 0)[0]] *= f
    return q


@pytest.mark.parametrize("uneven", [False, True])
@pytest.mark.parametrize("L,bc", [(2, PBC), (3, PBC), (4, PBC), (3, FREE), (4, FREE)])
@pytest.mark.parametrize("p", [0, 1, 2, 13, 15])
def test_fast_setup(p, L, bc, uneven):
    a = 5.3
    pos, q = uniform_system(90, a, seed=p + L)
    q = _uneven(q) if uneven else q
    g, o = mcfmm.Context(pos, q, a, L, p, bc=bc), O.System(pos, q, a, L, p, bc=bc)
    g.setup(mcfmm.SETUP_FMM)
    o.setup_fmm()
    for lev in range(2 if bc == PBC else 3, L + 1):
        _same(g.local(lev), o.local(lev), lev)
    if bc == PBC:
        # (p = 0: both sums of the neutral charges are rounding errors)
        K = o.KH()[0]
        assert np.max(np.abs(g.far()[0] - K)) <= ARR_TOL * max(np.max(np.abs(K)), np.max(np.abs(q)))
    _energies(g, o)
    g.close()


@pytest.mark.parametrize("uneven", [False, True])
@pytest.mark.parametrize("p,L,bc", [(0, 2, PBC), (1, 3, PBC), (2, 4, PBC), (15, 2, PBC), (14, 3, FREE), (15, 4, PBC)])
def test_multipole_setup(p, L, bc, uneven):
    a = 5.3
    pos, q = uniform_system(90, a, seed=p + L)
    q = _uneven(q) if uneven else q
    g, o = mcfmm.Context(pos, q, a, L, p, bc=bc), O.System(pos, q, a, L, p, bc=bc)
    g.setup(mcfmm.SETUP_MULTIPOLE)
    o.setup_multipole()
    for lev in range(2 if bc == PBC else 3, L + 1):
        _same(g.multipole(lev), o.multipole(lev), lev)
    _energies(g, o)
    g.close()


@pytest.mark.parametrize("L,bc,mode", [(2, PBC, mcfmm.SETUP_P2L), (3, PBC, mcfmm.SETUP_P2L), (3, FREE, mcfmm.SETUP_FMM),
                                       (3, PBC, mcfmm.SETUP_MULTIPOLE)])
def test_near_pairs_by_particle_count(L, bc, mode):
    """cells of 0..65 particles side by side: every split of a warp's lanes"""
    counts = [1, 2, 3, 4, 5, 8, 9, 15, 16, 17, 18, 31, 32, 33, 34, 36, 37, 40, 41, 47, 48, 49, 0, 63, 64, 65]
    a, nL = 6.7, 1 << (L - 1)
    rng = np.random.default_rng(L)
    cells = np.stack(np.meshgrid(*[np.arange(nL)] * 3, indexing="ij"), -1).reshape(-1, 3)
    per = [counts[i % len(counts)] for i in rng.permutation(max(len(cells), len(counts)))][:len(cells)]
    if sum(per) % 2:
        per[int(np.argmax(per))] -= 1
    pos = np.concatenate([(c + rng.uniform(0.001, 0.999, (k, 3))) * (a / nL) for c, k in zip(cells, per)])
    q = np.where(np.arange(len(pos)) % 2 == 0, 1.0, -1.0)
    g, o = mcfmm.Context(pos, q, a, L, 6, bc=bc), O.System(pos, q, a, L, 6, bc=bc)
    g.setup(mode)
    {mcfmm.SETUP_P2L: o.setup, mcfmm.SETUP_FMM: o.setup_fmm, mcfmm.SETUP_MULTIPOLE: o.setup_multipole}[mode]()
    _energies(g, o)
    g.close()


@pytest.mark.parametrize("d", [1e-19, 1e-15, 1e-12, 1e-9, 1e-6, 9e-4, 1.1e-3])
@pytest.mark.parametrize("where", ["corner", "face", "middle"])
def test_near_pair_of_any_distance(d, where):
    """two charges d finest cells apart: at the box's corner, where their
    coordinates have bits below 2^-62 of the box, across a periodic face and
    in a cell"""
    a, L = 6.4, 4
    w = a / (1 << (L - 1))
    pos, q = uniform_system(60, a, seed=2)
    i, j = int(np.argmax(q)), int(np.argmin(q))
    pos[i] = {"corner": [0.0, 0.0, 0.0], "face": [0.0, 1.3, 2.9], "middle": [1.1, 1.3, 2.9]}[where]
    step = np.array([0.6, 0.0, 0.8]) * d * w if where == "corner" else np.array([max(d, 1e-4) * w, 0.0, 0.0])
    pos[j] = (pos[i] + (-step if where == "face" else step)) % a
    g, o = mcfmm.Context(pos, q, a, L, 5), O.System(pos, q, a, L, 5)
    g.setup(mcfmm.SETUP_FMM)
    o.setup_fmm()
    assert np.isfinite(o.energy())
    _energies(g, o)
    g.close()


def test_fresh_energy_after_moves():
    a, L, p = 8.0, 3, 9
    pos, q = uniform_system(300, a, seed=3)
    g = mcfmm.Context(pos, q, a, L, p)
    g.setup()
    g.run(400, seed=5, beta=0.7, half_width=0.9)
    o = O.System(g.positions(), q, a, L, p)
    o.setup()
    assert abs(g.energy_fresh() - o.energy()) <= E_TOL * max(1.0, abs(o.energy()))
    g.close()
