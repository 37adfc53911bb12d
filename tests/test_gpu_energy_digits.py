"""Setup energies against extended precision, together with those of the FP64
kernel on the same charges (forced by two charges of 2^-10).  An energy has one
rounding error, so the root mean square over 24 systems counts; that of 24
values scatters by 15 %, the ratio of two by 20 %: the bound is 1.2 times the
FP64 error (a single running sum over a charge's near pairs, each pair counted
once, is 1.4 to 1.9 times off).
"""
import numpy as np
import pytest

from paper_2006_16622_gb300 import mcfmm
from paper_2006_16622_gb300.workloads import uniform_system
from test_gpu_level_digits import _exact
from test_gpu_multipole_digits import _multipoles

pytestmark = pytest.mark.gpu

LD = np.longdouble


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    mcfmm.load()


def _energy(pos, q, a, p):
    """U of the method at 3 levels in free space"""
    cells = np.stack(np.meshgrid(*[np.arange(4)] * 3, indexing="ij"), -1).reshape(-1, 3)
    W = np.concatenate([[1] + [2] * (2 * n) for n in range(p + 1)])
    u = np.sum(W * _exact(pos, q, a, 3, p, cells, True) * _multipoles(pos, q, a, 4, p)) / 2
    c, x = np.floor(pos * (4 / a)).astype(int), pos.astype(LD)
    i, j = np.nonzero(np.triu(np.all(np.abs(c[:, None] - c[None]) <= 1, -1), 1))
    d = x[i] - x[j]
    return u + np.sum(q[i] * q[j] / np.sqrt(np.sum(d * d, 1)))


def test_no_further_off_than_in_fp64():
    n, a, p = 1200, 10.0, 4
    err = {}
    for s in range(24):
        pos, q = uniform_system(n, a, seed=400 + s)
        qq = q.copy()
        qq[int(np.argmax(q))] = 2.0 ** -10
        qq[int(np.argmin(q))] = -2.0 ** -10
        for form, x in (("fixed", q), ("fp64", qq)):
            ref = _energy(pos, x, a, p)
            c = mcfmm.Context(pos, x, a, 3, p, bc=mcfmm.BC_FREE)
            for mode in (mcfmm.SETUP_P2L, mcfmm.SETUP_MULTIPOLE):
                c.setup(mode)
                err.setdefault((form, mode), []).append(float(LD(c.energy()) - ref))
            c.close()
    rms = {k: np.sqrt(np.mean(np.square(v))) for k, v in err.items()}
    for mode in (mcfmm.SETUP_P2L, mcfmm.SETUP_MULTIPOLE):
        assert rms["fixed", mode] <= 1.2 * rms["fp64", mode], rms
