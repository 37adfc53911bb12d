"""Expansions of the fast setup degree by degree against translations of the
charges' exact multipoles in extended precision, together with the FP64
translations of the same system (forced by two charges of 2^-10): the
fixed-point ones are no further off in any degree.  The box of side 1 lets the
high degrees outweigh the others; in the last system half of the charges lie
in one cell, so that cells beside it differ a thousandfold.

In units of a degree's norm both errors are averages over some cells, most of
it from the same matrices; they are compared with a factor 1.5 for their
scatter (degree 0: one coefficient a cell, left to the absolute bound) and
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


def _multipoles(pos, q, cells, nl, a, p):
    """sum q conj R_n^m(r - centre) of some cells in cell units, [cell][n][m]"""
    c = np.floor(pos * (nl / a)).astype(int)
    x, y, z = (pos.astype(LD) * (nl / LD(a)) - (c + LD(0.5))).T
    r2 = x * x + y * y + z * z
    index = {tuple(v): i for i, v in enumerate(cells)}
    at = np.array([index.get(tuple(v), -1) for v in c])
    x, y, z, r2, q, at = (v[at >= 0] for v in (x, y, z, r2, q, at))
    out = np.zeros((len(cells), p + 1, p + 1), np.clongdouble)
    cr, ci = np.ones(len(q), LD), np.zeros(len(q), LD)
    for m in range(p + 1):
        if m:
            cr, ci = (cr * x - ci * y) / (2 * m), (cr * y + ci * x) / (2 * m)
        b, g = (0 * cr, 0 * ci), (cr, ci)
        for n in range(m, p + 1):
            if n > m:
                den = LD((n + m) * (n - m))
                b, g = g, tuple(((2 * n - 1) * z * g[i] - r2 * b[i]) / den for i in (0, 1))
            np.add.at(out[:, n, m], at, q * (g[0] - 1j * g[1]))
    return out


def _irregular(o, lmax):
    x, y, z = (LD(v) for v in o)
    i2 = 1 / (x * x + y * y + z * z)
    out = np.zeros((lmax + 1, lmax + 1), np.clongdouble)
    c = np.clongdouble(np.sqrt(i2))
    for m in range(lmax + 1):
        if m:
            c = c * ((2 * m - 1) * i2 * (x + 1j * y))
        b, g = 0 * c, c
        for n in range(m, lmax + 1):
            if n > m:
                b, g = g, i2 * ((2 * n - 1) * z * g - ((n - 1) ** 2 - m * m) * b)
            out[n, m] = g
    return out


def _exact(pos, q, a, level, p, targets, free):
    """L_j^k of the target cells, real layout"""
    nl = 1 << (level - 1)
    lists = []
    for t in targets:
        r = [range(-2 - v, 4 - v) for v in t & 1]
        for o in ((i, j, k) for i in r[0] for j in r[1] for k in r[2]):
            s = t + np.array(o)
            if max(map(abs, o)) > 1 and not (free and np.any((s < 0) | (s >= nl))):
                lists.append((tuple(t), o, tuple(s % nl)))
    cells = sorted({s for _, _, s in lists})
    K = _multipoles(pos, q, np.array(cells), nl, a, p)
    sign = lambda m: -1 if m & 1 else 1
    full = np.stack([K[:, n, m] if m >= 0 else sign(m) * np.conj(K[:, n, -m])
                     for n in range(p + 1) for m in range(-n, n + 1)], 1)
    full = dict(zip(cells, full))
    rows = [(j, k) for j in range(p + 1) for k in range(j + 1)]
    L = {tuple(t): np.zeros(len(rows), np.clongdouble) for t in targets}
    by = {}
    for t, o, s in lists:
        by.setdefault(o, []).append((t, s))
    for o, pairs in by.items():
        I = _irregular(o, 2 * p)
        I = np.concatenate([I, [[sign(m) * np.conj(v) for m, v in enumerate(r)] for r in I]], 1)  # column w + m: order -m
        w = 2 * p + 1
        n = np.repeat(np.arange(p + 1), 2 * np.arange(p + 1) + 1)
        m = np.concatenate([np.arange(-v, v + 1) for v in range(p + 1)])
        j, k = (np.array(v)[:, None] for v in zip(*rows))
        km = k + m
        T = (1 - 2 * (n & 1)) * I[j + n, np.where(km >= 0, km, w - km)]
        for t, s in pairs:
            L[t] += np.conj(T @ full[s])
    out = np.zeros((len(targets), (p + 1) ** 2), LD)
    wl = LD(a) / nl
    for i, t in enumerate(targets):
        for (j, k), v in zip(rows, L[tuple(t)]):
            f = wl ** (-j - 1) / np.sqrt(LD(math.factorial(j - k)) * LD(math.factorial(j + k)))
            c = j * j + (2 * k - 1 if k else 0)
            out[i, c] = v.real * f
            if k:
                out[i, c + 1] = v.imag * f
    return out


def _by_degree(got, ref, p):
    e = got.astype(LD) - ref
    return np.array([float(np.sqrt(np.sum(e[:, n * n:(n + 1) ** 2] ** 2) / np.sum(ref[:, n * n:(n + 1) ** 2] ** 2))) for n in range(p + 1)])


@pytest.mark.parametrize("n,a,L,p,bc,dense", [(1200, 1.0, 3, 4, mcfmm.BC_PBC, False), (1200, 1.0, 3, 6, mcfmm.BC_FREE, False),
                                              (1300, 23.7, 3, 7, mcfmm.BC_FREE, False), (1400, 23.7, 3, 8, mcfmm.BC_PBC, False),
                                              (1500, 1.0, 3, 9, mcfmm.BC_FREE, False), (1600, 1.0, 3, 12, mcfmm.BC_PBC, False),
                                              (1600, 23.7, 3, 15, mcfmm.BC_PBC, False), (3000, 1.0, 4, 8, mcfmm.BC_FREE, True)])
def test_no_degree_further_off_than_in_fp64(n, a, L, p, bc, dense):
    pos, q = uniform_system(n, a, seed=n + p)
    nl = 1 << (L - 1)
    if dense:
        k = n // 2
        pos[:k] = (0.001 + 0.99 * np.random.default_rng(p).uniform(0.0, 1.0, (k, 3))) * (a / nl)
        q[:k] = 1.0
    qq = q.copy()
    i, j = len(q) - 1 - int(np.argmax(q[::-1])), int(np.argmin(q))
    qq[i] = 2.0 ** -10
    qq[j] = -2.0 ** -10
    # cells of every parity, all within reach of the dense one
    cells = np.stack(np.meshgrid(*[np.arange(4)] * 3, indexing="ij"), -1).reshape(-1, 3)
    targets = cells[(cells.max(1) >= 2)][::3 if p < 12 else 9]
    flat = (targets[:, 0] * nl + targets[:, 1]) * nl + targets[:, 2]
    err = {}
    for form, x in (("fixed", q), ("fp64", qq)):
        c = mcfmm.Context(pos, x, a, L, p, bc=bc)
        c.setup(mcfmm.SETUP_FMM)
        err[form] = _by_degree(c.local(L)[flat], _exact(pos, x, a, L, p, targets, bc == mcfmm.BC_FREE), p)
        c.close()
    f, d = err["fixed"], err["fp64"]
    assert f[0] <= 2.0 ** -50
    assert np.all(f[1:] <= np.maximum(1.5 * d[1:], 2.0 ** -51)), (f, d)
