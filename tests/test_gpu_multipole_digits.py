"""Multipoles of the finest level against sums in extended precision: the cells'
centres enter unrounded (box side with a full mantissa, many cells an axis).

Bound: a term of degree n is a product of n displacements, each off by 2^-53
of itself, and about as many roundings; 2^-53 (2 n + 4) for n = 8 is 2.2e-15
for every term, and the level's norm averages over thousands of them.
"""
import math

import numpy as np
import pytest

from paper_2006_16622_gb300 import mcfmm
from paper_2006_16622_gb300.workloads import uniform_system

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


def _multipoles(pos, q, a, nl, p):
    """M_n^m = sum q r^n Y_n^-m about the cells' centres, real layout"""
    c = np.floor(pos * (nl / a)).astype(int)
    x, y, z = (pos.astype(LD) - (c + LD(0.5)) * (LD(a) / nl)).T
    r2 = x * x + y * y + z * z
    cell = (c[:, 0] * nl + c[:, 1]) * nl + c[:, 2]
    out = np.zeros((nl ** 3, (p + 1) ** 2), LD)
    cr, ci = np.ones(len(q), LD), np.zeros(len(q), LD)
    for m in range(p + 1):
        if m:
            cr, ci = (cr * x - ci * y) / (2 * m), (cr * y + ci * x) / (2 * m)
        b, g = (0 * cr, 0 * ci), (cr, ci)
        for n in range(m, p + 1):
            if n > m:
                den = LD((n + m) * (n - m))
                b, g = g, tuple(((2 * n - 1) * z * g[i] - r2 * b[i]) / den for i in (0, 1))
            s = np.sqrt(LD(math.factorial(n - m)) * LD(math.factorial(n + m)))
            k = n * n + (2 * m - 1 if m else 0)
            np.add.at(out[:, k], cell, q * g[0] * s)
            if m:
                np.add.at(out[:, k + 1], cell, -q * g[1] * s)
    return out


def test_finest_level():
    n, a, L, p = 4000, 34.19951893353394, 5, 8
    pos, q = uniform_system(n, a, seed=3)
    c = mcfmm.Context(pos, q, a, L, p, bc=mcfmm.BC_FREE)
    c.setup(mcfmm.SETUP_MULTIPOLE)
    ref = _multipoles(pos, q, a, 1 << (L - 1), p)
    err = np.sqrt(float(np.sum((c.multipole(L).astype(LD) - ref) ** 2) / np.sum(ref ** 2)))
    c.close()
    assert err <= 2.2e-15, err
