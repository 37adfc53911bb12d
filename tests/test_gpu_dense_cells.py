"""Energy of systems whose charges gather in a few finest cells: the near pairs
of such cells are shared by many warps.

Energies against the oracle to 1e-10 as in the other parity tests, and the time
of a fresh energy against that of the per-particle FP64 kernel (which a context
with one charge of a very different size takes) on the same positions.
"""
import time

import numpy as np
import pytest

import oracle as O
from paper_2006_16622_gb300 import mcfmm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    mcfmm.load()


def _system(counts, a, L, others, seed):
    """counts: {(i, j, k) of a finest cell: charges}, others anywhere"""
    rng = np.random.default_rng(seed)
    w = a / (1 << (L - 1))
    pos = [(np.array(c) + rng.uniform(0.001, 0.999, (k, 3))) * w for c, k in counts.items()]
    pos = np.concatenate(pos + [rng.uniform(0.0, a, (others, 3))])
    pos = pos[:len(pos) // 2 * 2]
    return pos, np.where(np.arange(len(pos)) % 2 == 0, 1.0, -1.0)


@pytest.mark.parametrize("bc", [mcfmm.BC_PBC, mcfmm.BC_FREE])
@pytest.mark.parametrize("L,counts", [
    (3, {(1, 1, 1): 300}), (3, {(0, 0, 0): 129, (3, 3, 3): 257}), (3, {(0, 1, 2): 128, (0, 1, 3): 260, (0, 2, 3): 127}),
    (2, {(0, 0, 0): 400, (1, 0, 1): 130}), (4, {(7, 7, 7): 385, (7, 7, 6): 1, (0, 0, 0): 200})])
def test_energy(L, counts, bc):
    a = 6.5
    pos, q = _system(counts, a, L, 60, L)
    g, o = mcfmm.Context(pos, q, a, L, 6, bc=bc), O.System(pos, q, a, L, 6, bc=bc)
    g.setup()
    o.setup()
    for e in (g.energy(), g.energy_fresh()):
        assert abs(e - o.energy()) <= 1e-10 * max(1.0, abs(o.energy()))
    g.close()


def test_time_of_a_dense_cell():
    import torch
    a, L = 40.0, 5
    pos, q = _system({(5, 5, 5): 4000}, a, L, 4000, 1)
    t = []
    for even in (True, False):
        q = q.copy()
        if not even:
            q[-1] = 1e-6
        c = mcfmm.Context(pos, q, a, L, 8, bc=mcfmm.BC_FREE)
        c.setup()
        c.energy_fresh()
        best = 1e9
        for _ in range(5):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            c.energy_fresh()
            best = min(best, time.perf_counter() - t0)
        t.append(best)
        c.close()
    # (one warp for all pairs of the dense cell took 79 times as long)
    assert t[0] <= 5.0 * t[1], t
