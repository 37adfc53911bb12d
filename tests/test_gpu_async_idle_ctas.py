"""Barrier-free chains with so few items that whole CTAs own none: such a CTA
only polls and decides, nothing it does is waited for by an item, and it still
has to stay within the four-deep rings (few cells and p = 0 up to a grid that
is fully used; every SM, and fewer).

dE against the schedule with a grid barrier per phase: 1e-10 max(1, |dE|), the
bound of the other parity tests; decisions equal.
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


@pytest.mark.parametrize("ctas", [0, 40])
@pytest.mark.parametrize("n,a,L,p,bc", [(16, 3.0, 2, 0, mcfmm.BC_PBC), (16, 3.0, 2, 0, mcfmm.BC_FREE),
                                        (40, 5.0, 2, 3, mcfmm.BC_PBC), (126, 7.0, 3, 1, mcfmm.BC_FREE),
                                        (900, 9.0, 4, 7, mcfmm.BC_PBC)])
def test_replay_equals_plain_schedule(n, a, L, p, bc, ctas):
    pos, q = uniform_system(n, a, seed=n)
    ctx = {}
    for s in (mcfmm.SCHEDULE_ASYNC, mcfmm.SCHEDULE_PLAIN):
        ctx[s] = mcfmm.Context(pos, q, a, L, p, bc=bc)
        ctx[s].setup()
        ctx[s].set_schedule(s)
        ctx[s].set_ctas(ctas)
    for seed in range(8):
        r = {s: c.run(400, seed=seed, beta=0.7, half_width=0.9, log=True) for s, c in ctx.items()}
        x, y = r[mcfmm.SCHEDULE_ASYNC], r[mcfmm.SCHEDULE_PLAIN]
        assert np.array_equal(x["acc"], y["acc"]) and np.array_equal(x["j"], y["j"])
        f = np.isfinite(y["dE"])
        assert np.array_equal(f, np.isfinite(x["dE"]))
        assert np.all(np.abs(x["dE"][f] - y["dE"][f]) <= 1e-10 * np.maximum(1.0, np.abs(y["dE"][f])))
