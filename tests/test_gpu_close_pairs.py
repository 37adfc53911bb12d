"""One pair of charges a small part of a finest cell apart, anywhere in a box
whose side is no power of two, and at its lower corner, where coordinates have
more bits than a fraction of the box holds: the energy is q q' / r.

Bound: each coordinate is rounded down by less than 2 units of 2^-60 of a cell
and a pair closer than 2^-7 of a cell in every component takes its distance
from the coordinates, so a difference is off by sqrt(3) 2^-52 of the distance
at most; the rest is a few roundings.  2^-50 in all.
"""
from fractions import Fraction
from math import isqrt

import numpy as np
import pytest

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


def _inverse_distance(r, s):
    d2 = sum((Fraction(float(x)) - Fraction(float(y))) ** 2 for x, y in zip(r, s))
    return Fraction(1 << 200, isqrt(int(d2 * (1 << 400))))


@pytest.mark.parametrize("L", [3, 6])
@pytest.mark.parametrize("where", ["corner", "anywhere"])
def test_energy_of_a_close_pair(L, where):
    a = 46.4
    w = a / (1 << (L - 1))
    rng = np.random.default_rng(L)
    worst = 0
    for d in 2.0 ** -np.linspace(1.0, 14.0, 27):
        u = rng.normal(size=3)
        step = d * w * u / np.linalg.norm(u)
        base = np.abs(step) * rng.uniform(1.0, 1.3, 3) if where == "corner" else rng.uniform(w, a - w, 3)
        pos = np.array([base, base + step])
        if where == "corner":
            pos = np.abs(pos)
        q = np.array([1.5, -1.25])
        c = mcfmm.Context(pos, q, a, L, 0, bc=mcfmm.BC_FREE)
        c.setup()
        exact = Fraction(float(q[0])) * Fraction(float(q[1])) * _inverse_distance(*pos)
        worst = max(worst, abs(Fraction(c.energy()) / exact - 1))
        c.close()
    assert worst <= Fraction(1, 2 ** 50), float(worst)
