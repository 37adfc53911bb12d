"""What a user of this framework has it do, as cases to be timed.

The framework runs Metropolis-Hastings Monte Carlo of charged particles with
the multilevel local-expansion electrostatics method.  A program creates a
context for its system, sets it up (Alg. L.3, its fast variant, or the
multipole method), and then either proposes and accepts its own moves one by
one or lets the library run whole chains, one system or many at a time.  The
cases cover each of these calls over the sizes of the repository's own
workloads (N = 1e3 .. 1e6, 3 to 6 levels, expansion orders 6 .. 15, periodic
and free space, FP64 and FP32-eval, with and without Lennard-Jones).

exact() restates the method with plain torch in 64 bits: truncated Legendre
series (the addition theorem) for the energy changes, spherical harmonics and
the translation theorem for the expansions.
"""
import math

import numpy as np
import torch

from paper_2006_16622_gb300 import mcfmm
from paper_2006_16622_gb300.workloads import (NACL_BETA, NACL_LJ_CUTOFF, NACL_LJ_EPS, NACL_LJ_SIGMA,
                                              batched_systems, nacl_full_mc_system, uniform_system)

MODES = {"p2l": mcfmm.SETUP_P2L, "fmm": mcfmm.SETUP_FMM, "multipole": mcfmm.SETUP_MULTIPOLE}
RHO = 0.1  # density of the uniform workloads


def listed():
    return [
        # the user loop of the paper's interface on the SMALL workload: every
        # proposed move one synchronous propose(), then accept() if taken;
        # the smallest calls, latency only
        dict(name="moves-1e3", kind="moves", n=1000, levels=3, p=8, bc="pbc", moves=16),
        # the SMALL workload as a chain run by the library, decisions logged
        dict(name="chain-1e3", kind="chain", n=1000, levels=3, p=8, bc="pbc", prec="fp64", mode="p2l", steps=1000, h=0.5),
        # the LARGE workload (N = 1e5, p = 12), the headline chain
        dict(name="chain-1e5", kind="chain", n=100000, levels=5, p=12, bc="pbc", prec="fp64", mode="p2l", steps=2000, h=0.3),
        # the HUGE workload in the FP32-eval form
        dict(name="chain32-1e6", kind="chain", n=1000000, levels=6, p=12, bc="pbc", prec="fp32", mode="fmm", steps=2000, h=0.3),
        # the paper's full Monte Carlo setting: 46^3 NaCl ions, p = 11,
        # Lennard-Jones term, low acceptance, ~190 ions in a finest cell
        dict(name="nacl-46", kind="nacl", m=46, levels=4, p=11, steps=2000),
        # 64 independent chains of uneven N in one launch
        dict(name="batch-64", kind="batch", chains=64, n_lo=1000, n_hi=50000, p=10, prec="fp64", steps=300),
        # a new system from host arrays to its first moves: what starting a
        # run, or each replica of a scan, costs
        dict(name="start-1e4", kind="start", n=10000, levels=4, p=10, mode="p2l", steps=200),
        # a small ragged free-space system at the highest order
        dict(name="setup-free", kind="setup", n=1778, levels=4, p=15, bc="free", dip="tinfoil", mode="p2l"),
        # Alg. L.3 on the LARGE workload: the default setup, and the re-setup
        # that the FP32-eval form repeats during a run
        dict(name="setup-1e5", kind="setup", n=100000, levels=5, p=12, bc="pbc", dip="tinfoil", mode="p2l"),
        # the fast setup of the HUGE workload
        dict(name="setup-fmm-1e6", kind="setup", n=1000000, levels=6, p=12, bc="pbc", dip="tinfoil", mode="fmm"),
        # the multipole method's setup at an odd order, vacuum surroundings
        dict(name="setup-mm-3e4", kind="setup", n=31622, levels=5, p=11, bc="pbc", dip="vacuum", mode="multipole"),
        # one level's expansions from the caller's own device buffers
        dict(name="level-1e5", kind="level", n=100000, levels=5, level=4, p=12, bc="pbc"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _even(n):
    return n + n % 2


def _levels(rng, n, per_cell=20.0):
    """the workloads' level rule (about 20 charges in a finest cell), or one level fewer"""
    L = max(3, 1 + int(round(math.log(n / per_cell, 8))))
    return max(3, L - (rng.random() < 0.2))


def draw(rng):
    kind = rng.choice(["moves", "chain", "chain", "setup", "setup", "setup", "level", "start", "batch", "nacl"])
    p = rng.randint(6, 13)
    if kind == "moves":
        n = _even(_log(rng, 200, 100000))
        return dict(kind=kind, n=n, levels=_levels(rng, n), p=p, bc=rng.choice(["pbc", "pbc", "free"]), moves=rng.randint(4, 16))
    if kind == "chain":
        n = _even(_log(rng, 1000, 300000))
        return dict(kind=kind, n=n, levels=_levels(rng, n), p=p, bc="pbc", prec=rng.choice(["fp64", "fp32"]),
                    mode=rng.choice(["p2l", "fmm", "multipole"] if n < 60000 else ["fmm"]), steps=rng.randint(200, 2000),
                    h=round(rng.uniform(0.2, 0.5), 3))
    if kind == "setup":
        mode = rng.choice(["p2l", "fmm", "multipole"])
        n = _even(_log(rng, 1000, 400000 if mode == "fmm" else 60000))
        return dict(kind=kind, n=n, levels=_levels(rng, n), p=p if n > 20000 else rng.randint(6, 15), bc=rng.choice(["pbc", "pbc", "free"]),
                    dip=rng.choice(["tinfoil", "vacuum"]), mode=mode)
    if kind == "level":
        n = _even(_log(rng, 1000, 60000))
        L = _levels(rng, n)
        return dict(kind=kind, n=n, levels=L, level=rng.randint(3, L), p=p, bc=rng.choice(["pbc", "free"]))
    if kind == "start":
        n = _even(_log(rng, 1000, 40000))
        return dict(kind=kind, n=n, levels=_levels(rng, n), p=p, mode=rng.choice(["p2l", "fmm"]), steps=rng.randint(50, 500))
    if kind == "batch":
        return dict(kind=kind, chains=rng.randint(8, 48), n_lo=1000, n_hi=_log(rng, 4000, 30000), p=rng.randint(6, 11),
                    prec=rng.choice(["fp64", "fp32"]), steps=rng.randint(100, 300))
    return dict(kind="nacl", m=rng.choice([22, 26, 30, 34, 38, 42]), levels=4 if rng.random() < 0.5 else 3, p=rng.randint(8, 12), steps=rng.randint(300, 2000))


# ------------------------------------------------------------------ the path
def _box(n):
    return (n / RHO) ** (1.0 / 3.0)


def _bc(case):
    return mcfmm.BC_FREE if case.get("bc") == "free" else mcfmm.BC_PBC


def _prec(case):
    return mcfmm.FP32_EVAL if case.get("prec") == "fp32" else mcfmm.FP64


def _system(case, seed):
    pos, q = uniform_system(case["n"], _box(case["n"]), seed)
    return pos, q, _box(case["n"])


def _moves(case, seed, a):
    g = np.random.Generator(np.random.Philox(key=[0xCA5E, seed]))
    k = case["moves"]
    return g.integers(0, case["n"], size=k), g.uniform(-0.5, 0.5, (k, 3)), np.log(1.0 - g.random(k))


def _moved(r, d, a, free):
    """r + d wrapped into the box; free space: kept inside it"""
    x = r + d
    if free:
        return np.where((x >= 0.0) & (x < a), x, r)
    x = np.where(x < 0.0, x + a, x)
    return np.where(x >= a, x - a, x)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        ctxs = []
        for n, a, levels, i in batched_systems(case["chains"], case["n_lo"], case["n_hi"], RHO, 20.0, seed):
            pos, q = uniform_system(n, a, seed=1000 * seed + i)
            c = mcfmm.Context(pos, q, a, levels, case["p"], precision=_prec(case))
            c.setup(mcfmm.SETUP_FMM)
            ctxs.append(c)
        b = mcfmm.Batch(ctxs)
        b.tune(trial_steps=100, beta=1.0, half_width=0.3)
        return dict(case=case, batch=b, seeds=np.arange(case["chains"], dtype=np.uint64) + np.uint64(seed))
    if kind == "nacl":
        spacing = 153.2 / 46
        pos, q, a = nacl_full_mc_system(case["m"], spacing * case["m"], seed)
        c = mcfmm.Context(pos, q, a, case["levels"], case["p"])
        c.set_lj(NACL_LJ_EPS, NACL_LJ_SIGMA, min(NACL_LJ_CUTOFF, a / (1 << (case["levels"] - 1))))
        c.setup(mcfmm.SETUP_FMM)
        return dict(case=case, ctx=c, seed=seed)
    pos, q, a = _system(case, seed)
    if kind == "start":
        return dict(case=case, pos=pos, q=q, a=a, seed=seed)
    if kind == "level":
        dev = torch.device("cuda")
        nL = 1 << (case["levels"] - 1)
        cell = np.clip(np.floor(pos * (nL / a)).astype(np.int64), 0, nL - 1)
        cell = (cell[:, 0] * nL + cell[:, 1]) * nL + cell[:, 2]
        order = np.argsort(cell, kind="stable")
        part = torch.from_numpy(np.concatenate([pos, q[:, None]], 1)[order]).to(dev)
        start = torch.from_numpy(np.concatenate([[0], np.cumsum(np.bincount(cell, minlength=nL ** 3))]).astype(np.int32)).to(dev)
        out = torch.empty((8 ** (case["level"] - 1), (case["p"] + 1) ** 2), dtype=torch.float64, device=dev)
        torch.cuda.synchronize()
        return dict(case=case, part=part, start=start, out=out, a=a)
    dip = mcfmm.VACUUM if case.get("dip") == "vacuum" else mcfmm.TINFOIL
    c = mcfmm.Context(pos, q, a, case["levels"], case["p"], bc=_bc(case), dipole_bc=dip, precision=_prec(case))
    st = dict(case=case, ctx=c, seed=seed, a=a)
    if kind == "moves":
        c.setup()
        st.update(pos=pos.copy(), moves=_moves(case, seed, a))
    elif kind == "chain":
        c.setup(MODES[case["mode"]])
    return st


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "moves":
        c, pos, a = state["ctx"], state["pos"], state["a"]
        dEs = []
        for j, d, logu in zip(*state["moves"]):
            r = _moved(pos[j], d, a, case["bc"] == "free")
            dE = c.propose(j, r)
            dEs.append(dE)
            if dE <= 0.0 or logu < -dE:
                c.accept(j, r, dE)
                pos[j] = r
        return {"dE": np.array(dEs), "energy": np.array(c.energy()), "pos": pos.copy()}
    if kind == "chain":
        c = state["ctx"]
        r = c.run(case["steps"], state["seed"], beta=1.0, half_width=case["h"], log=True)
        return {"j": r["j"], "dE": r["dE"], "acc": r["acc"], "energy": np.array(r["energy"]), "pos": c.positions()}
    if kind == "nacl":
        c = state["ctx"]
        r = c.run(case["steps"], state["seed"], beta=NACL_BETA, half_width=0.25, log=True)
        return {"j": r["j"], "dE": r["dE"], "acc": r["acc"], "energy": np.array(r["energy"]), "pos": c.positions()}
    if kind == "batch":
        r = state["batch"].run(case["steps"], state["seeds"], beta=1.0, half_width=0.3)
        return {"energy": np.array([s["energy"] for s in r["stats"]]), "accepted": np.array([s["accepted"] for s in r["stats"]])}
    if kind == "start":
        c = mcfmm.Context(state["pos"], state["q"], state["a"], case["levels"], case["p"])
        c.setup(MODES[case["mode"]])
        e0 = c.energy()
        r = c.run(case["steps"], state["seed"], beta=1.0, half_width=0.3)
        out = {"e0": np.array(e0), "energy": np.array(r["energy"]), "accepted": r["accepted"], "pos": c.positions()}
        c.close()
        return out
    if kind == "level":
        rc = mcfmm.p2l_level_noalloc(state["part"].data_ptr(), state["start"].data_ptr(), case["n"], state["a"], case["levels"],
                                     case["level"], case["p"], _bc(case), state["out"].data_ptr(),
                                     torch.cuda.current_stream().cuda_stream)
        if rc != mcfmm.MC_OK:
            raise RuntimeError(f"p2l_level_noalloc: {rc}")
        return {"local": state["out"]}
    c = state["ctx"]
    c.setup(MODES[case["mode"]])
    get = c.multipole if case["mode"] == "multipole" else c.local
    K, H = c.far()
    return {"energy": np.array(c.energy()), "K": K, "H": H, "levels": [get(l) for l in range(2, case["levels"] + 1)]}


# ------------------------------------------------------- what it cannot avoid
def _eval_flops(p):
    """one expansion set (three-term recurrences) and its contraction"""
    return 3.0 * (p + 1) * (p + 2) + 2.0 * (p + 1) ** 2


def _setup_work(n, levels, p, free, mode):
    C, lev = (p + 1) ** 2, levels - (2 if free else 1)
    ncell = sum(8.0 ** (l - 1) for l in range(2, levels + 1))
    e = _eval_flops(p)
    occ = n / 8.0 ** (levels - 1)
    near = n * 27.0 * occ * 11.0
    if mode == "p2l":
        f = n * lev * 189.0 * e + n * lev * e + near
    elif mode == "fmm":
        f = n * lev * e + 189.0 * ncell * 2.0 * C * C + n * lev * e + near
    else:
        f = n * lev * e + n * lev * 189.0 * e + near
    return {"bytes": 32.0 * n + 8.0 * ncell * C + 16.0 * C, "flops": f}


def _step_work(n, levels, p, lev, acc):
    C, e = (p + 1) ** 2, _eval_flops(p)
    occ = n / 8.0 ** (levels - 1)
    prop = 2.0 * lev * e + 54.0 * occ * 11.0 + 6.0 * (p + 1) * (p + 2) + 2.0 * C * C + 4.0 * C + 297.0
    upd = 378.0 * lev * e + 4.0 * C
    return {"bytes": 16.0 * lev * C + 54.0 * occ * 32.0 + 8.0 * C * C + acc * (378.0 * lev * C * 16.0), "flops": prop + acc * upd}


def _times(w, k):
    return {"bytes": w["bytes"] * k, "flops": w["flops"] * k}


def _plus(a, b):
    return {"bytes": a["bytes"] + b["bytes"], "flops": a["flops"] + b["flops"]}


def work(case):
    kind = case["kind"]
    if kind == "batch":
        w = {"bytes": 0.0, "flops": 0.0}
        for n, a, levels, i in batched_systems(case["chains"], case["n_lo"], case["n_hi"], RHO, 20.0, 0):
            w = _plus(w, _times(_step_work(n, levels, case["p"], levels - 1, 0.9), case["steps"]))
        return w
    if kind == "nacl":
        n = case["m"] ** 3
        return _plus(_times(_step_work(n, case["levels"], case["p"], case["levels"] - 1, 0.35), case["steps"]),
                     {"bytes": 24.0 * n, "flops": 0.0})
    n, levels, p = case["n"], case["levels"], case["p"]
    free = case.get("bc") == "free"
    lev = levels - (2 if free else 1)
    if kind == "moves":
        return _times(_step_work(n, levels, p, lev, 0.9), case["moves"])
    if kind == "chain":
        return _plus(_times(_step_work(n, levels, p, lev, 0.9), case["steps"]), {"bytes": 24.0 * n, "flops": 0.0})
    if kind == "start":
        return _plus(_setup_work(n, levels, p, False, case["mode"]), _times(_step_work(n, levels, p, lev, 0.9), case["steps"]))
    if kind == "level":
        C = (p + 1) ** 2
        return {"bytes": 32.0 * n + 8.0 * C * 8.0 ** (case["level"] - 1), "flops": 189.0 * n * _eval_flops(p)}
    return _setup_work(n, levels, p, free, case["mode"])


# ------------------------------------- the same in 64 bits with plain torch
def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _cols(p):
    return [(n, m) for n in range(p + 1) for m in range(n + 1)]


def _norm(n, m):
    return math.sqrt(math.factorial(n - m) / math.factorial(n + m))


def _legendre(p, x, y, z, reg):
    """{(n, m): Y_n^m r^n} (reg) or {(n, m): Y_n^m / r^(n+1)} as (re, im),
    m >= 0, Y_n^m = sqrt((n-m)!/(n+m)!) P_n^m e^(i m phi), no Condon-Shortley phase"""
    r2 = x * x + y * y + z * z
    if reg:
        s, u, v, w = r2, x, y, z
        cur = (torch.ones_like(x), torch.zeros_like(x))
    else:
        s = 1.0 / r2
        u, v, w = x * s, y * s, z * s
        cur = (torch.sqrt(s), torch.zeros_like(x))
    for m in range(p + 1):
        if m:  # P_m^m = (2m-1) sin P_{m-1}^{m-1}, normalised
            f = (2 * m - 1) / math.sqrt((2 * m - 1) * 2 * m)
            cur = (f * (cur[0] * u - cur[1] * v), f * (cur[0] * v + cur[1] * u))
        b = None
        a = cur
        yield (m, m), a
        for n in range(m + 1, p + 1):
            d = math.sqrt((n - m) * (n + m))
            A, B = (2 * n - 1) / d, math.sqrt((n - 1 - m) * (n - 1 + m)) / d
            nxt = tuple(A * w * a[i] - (B * s * b[i] if b is not None else 0.0) for i in (0, 1))
            b, a = a, nxt
            yield (n, m), a


def _idx(n, m):
    return n * n + (2 * m - 1 if m else 0)


class _Cells:
    """the charges by cell of one level, padded with zero charges at the centre"""

    def __init__(self, pos, q, a, level, dev):
        self.nl = nl = 1 << (level - 1)
        self.w = a / nl
        c = torch.clamp(torch.floor(pos * (nl / a)).long(), 0, nl - 1)
        self.c3 = c
        cell = (c[:, 0] * nl + c[:, 1]) * nl + c[:, 2]
        order = torch.argsort(cell, stable=True)
        cnt = torch.bincount(cell, minlength=nl ** 3)
        first = torch.cumsum(cnt, 0) - cnt
        slot = torch.arange(len(q), device=dev) - first[cell[order]]
        cap = max(1, int(cnt.max()))
        g = torch.arange(nl, device=dev)
        self.ijk = torch.stack(torch.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)
        self.centre = (self.ijk.double() + 0.5) * self.w
        self.pos = self.centre[:, None, :].repeat(1, cap, 1)
        self.q = torch.zeros((nl ** 3, cap), dtype=torch.float64, device=dev)
        self.id = torch.full((nl ** 3, cap), -1, dtype=torch.long, device=dev)
        self.pos[cell[order], slot] = pos[order]
        self.q[cell[order], slot] = q[order]
        self.id[cell[order], slot] = order

    def at(self, t, o, free, a):
        """wrapped cells t + o, their image shifts, and which of them exist"""
        e = t + o
        src = e % self.nl
        ok = ((e == src).all(-1) if free else torch.ones(e.shape[:-1], dtype=torch.bool, device=e.device))
        return (src[..., 0] * self.nl + src[..., 1]) * self.nl + src[..., 2], (e - src).double() / self.nl * a, ok


def _lists(dev):
    """per parity class: the 189 offsets of the interaction list"""
    out = []
    for par in range(8):
        b = [(par >> 2) & 1, (par >> 1) & 1, par & 1]
        r = [range(-2 - v, 4 - v) for v in b]
        out.append(torch.tensor([(x, y, z) for x in r[0] for y in r[1] for z in r[2] if max(abs(x), abs(y), abs(z)) > 1], device=dev))
    return out


def _class(cells, par):
    i = cells.ijk
    return torch.nonzero(((i[:, 0] & 1) * 4 + (i[:, 1] & 1) * 2 + (i[:, 2] & 1)) == par)[:, 0]


def _chunks(total, row, most=1 << 24):
    step = max(1, most // max(1, row))
    return [(i, min(total, i + step)) for i in range(0, total, step)]


def _p2l(cells, p, free, a, lists):
    """Alg. L.3 of one level: L_n^m = sum q Y_n^-m / r^(n+1), real layout"""
    out = torch.zeros((cells.nl ** 3, (p + 1) ** 2), dtype=torch.float64, device=cells.q.device)
    for par in range(8):
        t = _class(cells, par)
        cap = cells.q.shape[1]
        for lo, hi in _chunks(len(t), 189 * cap):
            src, shift, ok = cells.at(cells.ijk[t[lo:hi]][:, None, :], lists[par][None], free, a)
            d = (cells.pos[src] + shift[:, :, None, :] - cells.centre[t[lo:hi]][:, None, None, :]).reshape(hi - lo, -1, 3)
            qq = (cells.q[src] * ok[:, :, None]).reshape(hi - lo, -1)
            d = torch.where(qq[..., None] == 0.0, torch.full_like(d, cells.w * 3), d)
            for (n, m), (re, im) in _legendre(p, d[..., 0].contiguous(), d[..., 1].contiguous(), d[..., 2].contiguous(), False):
                out[t[lo:hi], _idx(n, m)] = (qq * re).sum(-1)
                if m:
                    out[t[lo:hi], _idx(n, m) + 1] = -(qq * im).sum(-1)
    return out


def _p2m(cells, p):
    """multipoles M_n^m = sum q r^n Y_n^-m about every centre, real layout"""
    d = cells.pos - cells.centre[:, None, :]
    out = torch.zeros((cells.nl ** 3, (p + 1) ** 2), dtype=torch.float64, device=cells.q.device)
    for lo, hi in _chunks(len(d), d.shape[1]):
        e, qq = d[lo:hi], cells.q[lo:hi]
        for (n, m), (re, im) in _legendre(p, e[..., 0].contiguous(), e[..., 1].contiguous(), e[..., 2].contiguous(), True):
            out[lo:hi, _idx(n, m)] = (qq * re).sum(-1)
            if m:
                out[lo:hi, _idx(n, m) + 1] = -(qq * im).sum(-1)
    return out


def _complex(x, p):
    """real layout -> all m = -n..n, index n^2 + n + m"""
    out = torch.zeros(x.shape, dtype=torch.complex128, device=x.device)
    for n, m in _cols(p):
        v = torch.complex(x[..., _idx(n, m)], x[..., _idx(n, m) + 1]) if m else x[..., n * n].to(torch.complex128)
        out[..., n * n + n + m] = v
        out[..., n * n + n - m] = v.conj()
    return out


def _real(x, p):
    out = torch.zeros(x.shape, dtype=torch.float64, device=x.device)
    for n, m in _cols(p):
        v = x[..., n * n + n + m]
        out[..., _idx(n, m)] = v.real
        if m:
            out[..., _idx(n, m) + 1] = v.imag
    return out


def _m2l_matrices(p, S):
    """Greengard-Rokhlin translation: L_j^k = sum_nm T[j,k;n,m] M_n^m with
    S[..., l^2 + l + m] = Y_l^m / rho^(l+1) of the source offset, l <= 2p"""
    C = (p + 1) ** 2
    row, col, src, fac = [], [], [], []
    f = [float(math.factorial(i)) for i in range(4 * p + 1)]
    A = lambda n, m: (-1.0) ** n / math.sqrt(f[n - m] * f[n + m])  # noqa: E731
    for j in range(p + 1):
        for k in range(-j, j + 1):
            for n in range(p + 1):
                for m in range(-n, n + 1):
                    e = abs(k - m) - abs(k) - abs(m)
                    row.append(j * j + j + k)
                    col.append(n * n + n + m)
                    src.append((j + n) ** 2 + (j + n) + m - k)
                    fac.append((-1.0) ** (e // 2) * A(n, m) * A(j, k) / ((-1.0) ** n * A(j + n, m - k)))
    dev = S.device
    T = torch.zeros(S.shape[:-1] + (C, C), dtype=torch.complex128, device=dev)
    T[..., torch.tensor(row, device=dev), torch.tensor(col, device=dev)] = S[..., torch.tensor(src, device=dev)] * torch.tensor(fac, dtype=torch.float64, device=dev)
    return T


def _m2l(cells, p, M, free, a, lists):
    dev = M.device
    grid = torch.stack(torch.meshgrid(*[torch.arange(-3, 4, device=dev)] * 3, indexing="ij"), -1).reshape(-1, 3)
    far = grid.abs().max(-1).values > 1
    o = torch.where(far[:, None], grid, torch.full_like(grid, 2)).double() * cells.w
    S = torch.zeros((343, (2 * p + 1) ** 2), dtype=torch.complex128, device=dev)
    for (l, m), (re, im) in _legendre(2 * p, o[:, 0], o[:, 1], o[:, 2], False):
        S[:, l * l + l + m] = torch.complex(re, im)
        S[:, l * l + l - m] = torch.complex(re, -im)
    Mc = torch.cat([_complex(M, p), torch.zeros((1, M.shape[1]), dtype=torch.complex128, device=dev)])
    out = torch.zeros((len(M), M.shape[1]), dtype=torch.complex128, device=dev)
    byo = [[] for _ in range(343)]
    for par in range(8):
        t = _class(cells, par)
        for off in lists[par]:
            src, _, ok = cells.at(cells.ijk[t], off, free, a)
            byo[int(((off[0] + 3) * 7 + off[1] + 3) * 7 + off[2] + 3)].append((t, torch.where(ok, src, torch.full_like(src, len(M)))))
    for i, parts in enumerate(byo):
        if parts:
            T = _m2l_matrices(p, S[i])
            t, src = torch.cat([x[0] for x in parts]), torch.cat([x[1] for x in parts])
            out[t] += Mc[src] @ T.T
    return _real(out, p)


def _lattice(p, dev):
    """S_l^m = sum over integer v, max|v_i| >= 2, of Y_l^m(v)/|v|^(l+1), l <= 2p:
    Poisson summation of the harmonic polynomials (3 <= l < 20), split at 2,
    the 26 nearest images removed; direct sums above"""
    lmax = 2 * p
    S = torch.zeros((lmax + 1) ** 2, dtype=torch.complex128, device=dev)

    def grid(R):
        g = torch.arange(-R, R + 1, device=dev)
        v = torch.stack(torch.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)
        return v[v.abs().max(-1).values > 0]

    v, kv = grid(12), grid(9)
    r2, k2 = (v * v).sum(-1).double(), (kv * kv).sum(-1).double()
    near = v.abs().max(-1).values <= 1
    X = 2.0 * math.pi * r2
    Q, term, Qs = torch.erfc(torch.sqrt(X)), torch.sqrt(X) * torch.exp(-X) / (0.5 * math.sqrt(math.pi)), []
    for i in range(21):
        Qs.append(Q.clone())  # Q(i + 1/2, X)
        Q = Q + term
        term = term * X / (i + 1.5)
    rv = [v[:, i].double() for i in range(3)]
    for (l, m), (re, im) in _legendre(lmax, *rv, False):
        if l < 3:
            continue
        wgt = (Qs[l] if l < 20 else torch.ones_like(r2)) - near.double()
        S[l * l + l + m] += torch.complex((wgt * re).sum(), (wgt * im).sum())
    rk = [kv[:, i].double() for i in range(3)]
    for (l, m), (re, im) in _legendre(min(lmax, 19), *rk, True):
        if l < 3:
            continue
        wgt = math.pi ** (l - 0.5) / math.gamma(l + 0.5) * torch.exp(-math.pi * k2 / 2.0) / k2
        S[l * l + l + m] += torch.complex((wgt * re).sum(), (wgt * im).sum()) * (-1j) ** l
    for l in range(3, lmax + 1):
        for m in range(1, l + 1):
            S[l * l + l - m] = S[l * l + l + m].conj()
    return S


def _far_operator(p, a, dev):
    l = torch.tensor([l for l in range(2 * p + 1) for _ in range(2 * l + 1)], dtype=torch.float64, device=dev)
    return _m2l_matrices(p, _lattice(p, dev) * torch.pow(torch.tensor(a, dtype=torch.float64, device=dev), -(l + 1)))


def _box_multipole(pos, q, a, p):
    d = pos - 0.5 * a
    K = torch.zeros((p + 1) ** 2, dtype=torch.float64, device=pos.device)
    for (n, m), (re, im) in _legendre(p, d[:, 0].contiguous(), d[:, 1].contiguous(), d[:, 2].contiguous(), True):
        K[_idx(n, m)] = (q * re).sum()
        if m:
            K[_idx(n, m) + 1] = -(q * im).sum()
    return K


def _weights(p, dev):
    return torch.tensor([1.0 if k == n * n else 2.0 for n in range(p + 1) for k in range(n * n, (n + 1) ** 2)], dtype=torch.float64, device=dev)


def _exact_setup(case, seed, dev):
    pos_h, q_h, a = _system(case, seed)
    pos, q = torch.from_numpy(pos_h).to(dev), torch.from_numpy(q_h).to(dev)
    p, L, free, mode = case["p"], case["levels"], case["bc"] == "free", case["mode"]
    lists, C = _lists(dev), (p + 1) ** 2
    lmin = 3 if free else 2
    got, phi = [], torch.zeros_like(q)
    for l in range(2, L + 1):
        if l < lmin:
            got.append(torch.zeros((8 ** (l - 1), C), dtype=torch.float64, device=dev))
            continue
        cells = _Cells(pos, q, a, l, dev)
        cell = (cells.c3[:, 0] * cells.nl + cells.c3[:, 1]) * cells.nl + cells.c3[:, 2]
        if mode == "p2l":
            E = _p2l(cells, p, free, a, lists)
        else:
            E = _p2m(cells, p)
            if mode == "fmm":
                E = _m2l(cells, p, E, free, a, lists)
        got.append(E)
        if mode == "multipole":  # the listed cells' multipole expansions at every charge
            table = torch.stack(lists)
            par = (cells.c3[:, 0] & 1) * 4 + (cells.c3[:, 1] & 1) * 2 + (cells.c3[:, 2] & 1)
            for lo, hi in _chunks(len(q), 189):
                off = table[par[lo:hi]]
                src, shift, ok = cells.at(cells.c3[lo:hi][:, None, :], off, free, a)
                d = pos[lo:hi][:, None, :] - (cells.centre[src] + shift)
                d = torch.where(ok[..., None], d, torch.full_like(d, cells.w * 3))
                s = torch.zeros_like(d[..., 0])
                for (n, m), (re, im) in _legendre(p, d[..., 0].contiguous(), d[..., 1].contiguous(), d[..., 2].contiguous(), False):
                    Mr = E[:, _idx(n, m)][src]
                    s += Mr * re if m == 0 else 2.0 * (Mr * re - E[:, _idx(n, m) + 1][src] * im)
                phi[lo:hi] += (s * ok).sum(-1)
        else:
            d = pos - cells.centre[cell]
            for (n, m), (re, im) in _legendre(p, d[:, 0].contiguous(), d[:, 1].contiguous(), d[:, 2].contiguous(), True):
                Er = E[:, _idx(n, m)][cell]
                phi += Er * re if m == 0 else 2.0 * (Er * re - E[:, _idx(n, m) + 1][cell] * im)
    cells = _Cells(pos, q, a, L, dev)
    near = torch.zeros_like(cells.q)
    for k in range(27):
        off = torch.tensor([k // 9 - 1, (k // 3) % 3 - 1, k % 3 - 1], device=dev)
        src, shift, ok = cells.at(cells.ijk, off, free, a)
        cap = cells.q.shape[1]
        for lo, hi in _chunks(len(src), cap * cap, 1 << 25):
            d = cells.pos[lo:hi][:, :, None, :] - (cells.pos[src[lo:hi]] + shift[lo:hi][:, None, :])[:, None, :, :]
            d2 = (d * d).sum(-1)
            w = cells.q[src[lo:hi]][:, None, :] * ok[lo:hi, None, None]
            drop = (d2 == 0.0) | (w == 0.0)
            near[lo:hi] += torch.where(drop, torch.zeros_like(d2), w / torch.sqrt(torch.where(drop, torch.ones_like(d2), d2))).sum(-1)
    keep = cells.id >= 0
    phi[cells.id[keep]] += near[keep]
    U = 0.5 * (q * phi).sum()
    K = H = torch.zeros(C, dtype=torch.float64, device=dev)
    if not free:
        K = _box_multipole(pos, q, a, p)
        H = _real(_far_operator(p, a, dev) @ _complex(K, p), p)
        U = U + 0.5 * (_weights(p, dev) * K * H).sum()
        if case["dip"] == "tinfoil":
            D = (q[:, None] * pos).sum(0)
            U = U - 2.0 * math.pi / (3.0 * a ** 3) * (D * D).sum()
    return {"energy": np.array(float(U)), "K": K.cpu().numpy(), "H": H.cpu().numpy(), "levels": [g.cpu().numpy() for g in got]}


class _Direct:
    """dE of one move by the method's definition: Alg. 1 on the near cells, the
    order-p Legendre series of the listed charges, the periodic terms"""

    def __init__(self, pos, q, a, L, p, free, dev):
        self.pos, self.q = torch.from_numpy(pos).to(dev), torch.from_numpy(q).to(dev)
        self.a, self.L, self.p, self.free, self.dev = a, L, p, free, dev
        g = torch.arange(-1, 2, device=dev)
        self.nu = torch.stack(torch.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)
        if free:
            self.nu = torch.zeros((1, 3), dtype=torch.long, device=dev)
        else:
            self.R, self.W = _far_operator(p, a, dev), _weights(p, dev)
            self.K, self.D = _box_multipole(self.pos, self.q, a, p), (self.q[:, None] * self.pos).sum(0)

    def cell(self, x, l):
        nl = 1 << (self.L - 1)
        return torch.clamp(torch.floor(x * (nl / self.a)).long(), 0, nl - 1) >> (self.L - l)

    def potential(self, r, j):
        """near sum without particle j at zero shift (j < 0: with all) and the level series at r"""
        phi = torch.zeros((), dtype=torch.float64, device=self.dev)
        img = self.pos[None] + self.nu[:, None, :].double() * self.a
        done = torch.zeros(img.shape[:-1], dtype=torch.bool, device=self.dev)
        for l in range(self.L, (2 if self.free else 1), -1):
            nl = 1 << (l - 1)
            c, ci = self.cell(r, l), self.cell(self.pos, l)[None] + self.nu[:, None, :] * nl
            near = (ci - c).abs().max(-1).values <= 1
            if l == self.L:
                take = near.clone()
                if j >= 0:
                    take[(len(self.nu) - 1) // 2, j] = False
                d = img[take] - r
                qn = self.q[None].expand(len(self.nu), -1)[take]
                phi = phi + (qn / torch.sqrt((d * d).sum(-1))).sum()
                done = near
            inlist = ((ci >> 1) - (c >> 1)).abs().max(-1).values <= 1
            inlist = inlist & ~near
            s = img[inlist] - (c.double() + 0.5) * (self.a / nl)
            x = r - (c.double() + 0.5) * (self.a / nl)
            qs = self.q[None].expand(len(self.nu), -1)[inlist]
            s2 = (s * s).sum(-1)
            t = (s * x).sum(-1) / s2  # |x|/|s| cos
            u = (x * x).sum() / s2
            a0, a1 = torch.ones_like(t), t
            tot = a0 + (a1 if self.p > 0 else 0.0)
            for n in range(2, self.p + 1):
                a0, a1 = a1, ((2 * n - 1) * t * a1 - (n - 1) * u * a0) / n
                tot = tot + a1
            phi = phi + (qs * tot / torch.sqrt(s2)).sum()
        return phi

    def change(self, j, rn):
        r, q = self.pos[j], self.q[j]
        dE = q * (self.potential(rn, -1) - self.potential(r, j))
        d = rn - (r + self.nu.double() * self.a)
        dE = dE - q * q * (1.0 / torch.sqrt((d * d).sum(-1))).sum()
        if not self.free:
            dE = dE + q * q / self.a * (6.0 + 8.0 / math.sqrt(3.0) + 12.0 / math.sqrt(2.0))
            one = torch.stack([rn, r])
            dK = _box_multipole(one[:1], q[None], self.a, self.p) - _box_multipole(one[1:], q[None], self.a, self.p)
            H = _real(self.R @ _complex(self.K + 0.5 * dK, self.p), self.p)
            dE = dE + (self.W * dK * H).sum()
            Dn = self.D + q * (rn - r)
            dE = dE - 2.0 * math.pi / (3.0 * self.a ** 3) * ((Dn * Dn).sum() - (self.D * self.D).sum())
            self.last = (dK, Dn)
        return float(dE)

    def take(self, j, rn):
        if not self.free:
            self.K, self.D = self.K + self.last[0], self.last[1]
        self.pos[j] = rn


def _philox(c, k):
    c, k = list(c), list(k)
    for r in range(10):
        if r:
            k = [(k[0] + 0x9E3779B9) & 0xFFFFFFFF, (k[1] + 0xBB67AE85) & 0xFFFFFFFF]
        x, y = 0xD2511F53 * c[0], 0xCD9E8D57 * c[2]
        c = [(y >> 32) ^ c[1] ^ k[0], y & 0xFFFFFFFF, (x >> 32) ^ c[3] ^ k[1], x & 0xFFFFFFFF]
    return c


def _exact_energy(case, seed, dev):
    return _exact_setup(dict(case, kind="setup", dip="tinfoil", mode="p2l"), seed, dev)["energy"].item()


def _exact_moves(case, seed, dev):
    pos, q, a = _system(case, seed)
    free = case["bc"] == "free"
    D, dEs, e = _Direct(pos, q, a, case["levels"], case["p"], free, dev), [], _exact_energy(case, seed, dev)
    pos = pos.copy()
    for j, d, logu in zip(*_moves(case, seed, a)):
        r = _moved(pos[j], d, a, free)
        rt = torch.from_numpy(np.ascontiguousarray(r)).to(dev)
        dE = 0.0 if (r == pos[j]).all() else D.change(int(j), rt)
        dEs.append(dE)
        if dE <= 0.0 or logu < -dE:
            if not (r == pos[j]).all():
                D.take(int(j), rt)
            pos[j] = r
            e += dE
    return {"dE": np.array(dEs), "energy": np.array(e), "pos": pos}


def _exact_chain(case, seed, dev):
    pos, q, a = _system(case, seed)
    n, h = case["n"], case["h"]
    D, e = _Direct(pos, q, a, case["levels"], case["p"], False, dev), _exact_energy(case, seed, dev)
    pos, js, dEs, acc = pos.copy(), [], [], []
    key = (seed & 0xFFFFFFFF, seed >> 32)
    for s in range(case["steps"]):
        A, B = _philox((s, 0, 0, 0), key), _philox((s, 0, 0, 1), key)
        j = (A[0] * n) >> 32
        d = np.array([h * (2.0 * ((A[k] + 0.5) * 2.0 ** -32) - 1.0) for k in (1, 2, 3)])
        u = ((B[0] >> 5) * 67108864.0 + (B[1] >> 6)) * 2.0 ** -53
        r = _moved(pos[j], d, a, False)
        rt = torch.from_numpy(np.ascontiguousarray(r)).to(dev)
        dE = D.change(j, rt)
        ok = dE <= 0.0 or (u > 0.0 and math.log(u) < -dE)
        if ok:
            D.take(j, rt)
            pos[j] = r
            e += dE
        js.append(j)
        dEs.append(dE)
        acc.append(ok)
    return {"j": np.array(js, dtype=np.int64), "dE": np.array(dEs), "acc": np.array(acc, dtype=np.uint8), "energy": np.array(e), "pos": pos}


def exact(case, seed):
    dev = _dev()
    kind = case["kind"]
    with torch.no_grad():
        if kind == "setup":
            return _exact_setup(case, seed, dev)
        if kind == "level":
            pos, q, a = _system(case, seed)
            pos, q = torch.from_numpy(pos).to(dev), torch.from_numpy(q).to(dev)
            free = case["bc"] == "free"
            return {"local": _p2l(_Cells(pos, q, a, case["level"], dev), case["p"], free, a, _lists(dev))}
        if kind == "moves" and case["n"] <= 40000:
            return _exact_moves(case, seed, dev)
        if kind == "chain" and case["prec"] == "fp64" and case["mode"] == "p2l" and case["n"] <= 4000 and case["steps"] <= 1000:
            return _exact_chain(case, seed, dev)
        if kind == "start" and case["mode"] == "p2l" and case["n"] <= 20000:
            e0 = _exact_energy(dict(case, bc="pbc"), seed, dev)
            return {"e0": np.array(e0), "energy": None, "accepted": None, "pos": None}
    return None  # a replay of the other chains takes minutes in plain torch
