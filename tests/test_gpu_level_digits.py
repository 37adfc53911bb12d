"""Alg. L.3 expansions degree by degree against sums in extended precision,
together with those of the FP64 gather on the same charges (forced by one more
charge, 2^-10 of the others): the fixed-point sums are no further off in any
degree.

In units of a degree's norm both errors are averages over all cells; they are
compared with a factor 1.3 for their scatter (a degree has 2 n + 1 >= 3
coefficients in 8 or more cells, degree 0 is left to the absolute bound) and
with 2^-51, half a dozen roundings of the result, as what need not be beaten.
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


def _list(b):
    r = [range(-2 - v, 4 - v) for v in b]
    return np.array([(x, y, z) for x in r[0] for y in r[1] for z in r[2] if max(abs(x), abs(y), abs(z)) > 1])


def _exact(pos, q, a, level, p, targets, free):
    """L_n^m of the target cells, real layout"""
    nl = 1 << (level - 1)
    w = LD(a) / nl
    c = np.floor(pos * (nl / a)).astype(int)
    by = {}
    for i, k in enumerate(map(tuple, c)):
        by.setdefault(k, []).append(i)
    out = np.zeros((len(targets), (p + 1) ** 2), LD)
    for row, t in enumerate(targets):
        at, qs = [], []
        for e in t + _list(t & 1):
            s = e % nl
            ids = by.get(tuple(s), [])
            if ids and not (free and np.any(e != s)):
                at.append(pos[ids].astype(LD) + ((e - s) // nl).astype(LD) * LD(a))
                qs.append(q[ids])
        x, y, z = (np.concatenate(at) - (t + LD(0.5)) * w).T
        qs = np.concatenate(qs)
        i2 = 1 / (x * x + y * y + z * z)
        cr, ci = np.sqrt(i2), 0 * x
        for m in range(p + 1):
            if m:
                f = (2 * m - 1) * i2
                cr, ci = f * (cr * x - ci * y), f * (cr * y + ci * x)
            b, g = (0 * cr, 0 * ci), (cr, ci)
            for n in range(m, p + 1):
                if n > m:
                    b, g = g, tuple(i2 * ((2 * n - 1) * z * g[i] - ((n - 1) ** 2 - m * m) * b[i]) for i in (0, 1))
                s = np.sqrt(LD(math.factorial(n - m)) * LD(math.factorial(n + m)))
                k = n * n + (2 * m - 1 if m else 0)
                out[row, k] = np.sum(qs * g[0]) / s
                if m:
                    out[row, k + 1] = -np.sum(qs * g[1]) / s
    return out


def _by_degree(got, ref, p):
    e = got.astype(LD) - ref
    return np.array([float(np.sqrt(np.sum(e[:, n * n:(n + 1) ** 2] ** 2) / np.sum(ref[:, n * n:(n + 1) ** 2] ** 2))) for n in range(p + 1)])


@pytest.mark.parametrize("n,a,L,p,bc", [(1000, 31.0, 3, 10, mcfmm.BC_PBC), (1000, 1.0, 3, 7, mcfmm.BC_PBC),
                                        (1300, 23.0, 3, 12, mcfmm.BC_FREE)])
def test_no_degree_further_off_than_in_fp64(n, a, L, p, bc):
    pos, q = uniform_system(n, a, seed=n)
    free = bc == mcfmm.BC_FREE
    qq = q.copy()
    i, j = int(np.argmax(q)), int(np.argmin(q))
    qq[i] = 2.0 ** -10
    qq[j] = -2.0 ** -10
    levels = [3] if free else [2, 3]
    err = {}
    for form, x in (("fixed", q), ("fp64", qq)):
        c = mcfmm.Context(pos, x, a, L, p, bc=bc)
        c.setup(mcfmm.SETUP_P2L)
        for l in levels:
            nl = 1 << (l - 1)
            cells = np.stack(np.meshgrid(*[np.arange(nl)] * 3, indexing="ij"), -1).reshape(-1, 3)
            pick = np.arange(0, nl ** 3, 1 if l == 2 else 5)
            err[form, l] = _by_degree(c.local(l)[pick], _exact(pos, x, a, l, p, cells[pick], free), p)
        c.close()
    for l in levels:
        f, d = err["fixed", l], err["fp64", l]
        assert f[0] <= 2.0 ** -50
        assert np.all(f[1:] <= np.maximum(1.3 * d[1:], 2.0 ** -51)), (l, f, d)
