"""Performance cases of the library: what its users run, through the public entry points.

A case is a dict of plain values; prepare() makes its inputs and handles from
a seed, run() makes one pass, work() states what the pass cannot do without,
exact() gives the same outputs in 64-bit torch without the library.

Paths: "apply" (H x), "lanczos" (a fixed number of steps), "ground" (a solve
to a tolerance, with the vector), "reorth" (reorthogonalised Lanczos with the
vector), "tpq" (one canonical-TPQ step), "evolve" (one real-time step),
"spectrum" (dynamical structure factor of several wave numbers), "batch" (many
small ground states in one call).  Models: "spin" (S^z sector), "full" (all
2^N states), "hubbard".
"""
import functools
import math
import random

import numpy as np
import torch

from paper_2307_13222_gb300 import hphi

DTYPES = {"f32": torch.float32, "f64": torch.float64, "c64": torch.complex64, "c128": torch.complex128}


def listed():
    return [
        # one product of the 16-site chain (the smallest configured problem): latency
        dict(name="apply_chain16_f64", path="apply", model="spin", lattice="chain", lx=16, ly=1, n_up=8, n_dn=0,
             random_j=False, dtype="f64", nvec=1, beta=0.0),
        # the metric's own product: 4x8 square lattice, 601,080,390 states
        dict(name="apply_square8x4_f32", path="apply", model="spin", lattice="square", lx=8, ly=4, n_up=16, n_dn=0,
             random_j=False, dtype="f32", nvec=1, beta=0.0),
        # a request of the serving mix: random-coupling ladder, an odd magnetisation, accumulating product
        dict(name="apply_ladder14_f64", path="apply", model="spin", lattice="square", lx=14, ly=2, n_up=13, n_dn=0,
             random_j=True, dtype="f64", nvec=1, beta=0.5),
        # 4x4 Hubbard at half filling, U = 8
        dict(name="apply_hubbard4x4_f32", path="apply", model="hubbard", lattice="square", lx=4, ly=4, n_up=8,
             n_dn=8, random_j=False, dtype="f32", nvec=1, beta=0.0),
        # a run of Lanczos steps of the FP32-storage route at a size between the two
        dict(name="lanczos_square6x5_f32", path="lanczos", model="spin", lattice="square", lx=6, ly=5, n_up=15,
             n_dn=0, random_j=False, dtype="f32", steps=20),
        # a whole ground-state solve of a mid-size request
        dict(name="ground_chain20_f64", path="ground", model="spin", lattice="chain", lx=20, ly=1, n_up=10, n_dn=0,
             random_j=True, dtype="f64", tol=1e-12, check_every=4),
        # reorthogonalised Lanczos on the largest Hubbard ladder of the serving mix
        dict(name="reorth_hubbard7x2_f32", path="reorth", model="hubbard", lattice="square", lx=7, ly=2, n_up=7,
             n_dn=7, random_j=True, dtype="f32", steps=40),
        # the cTPQ benchmark's step: 2^26 states, 16 complex FP32 vectors
        dict(name="tpq_full26_c64x16", path="tpq", model="full", lattice="rrg", lx=26, ly=1, n_up=0, n_dn=0,
             random_j=True, dtype="c64", nvec=16, nmax=6, dtau=0.02),
        # the same step in FP64 at a size of everyday runs
        dict(name="tpq_full21_c128x16", path="tpq", model="full", lattice="ladder", lx=10, ly=2, n_up=0, n_dn=0,
             random_j=True, dtype="c128", nvec=16, nmax=6, dtau=0.02),
        # a Hubbard quench: one complex FP64 wave function
        dict(name="evolve_hubbard6x2_c128", path="evolve", model="hubbard", lattice="square", lx=6, ly=2, n_up=6,
             n_dn=6, random_j=False, dtype="c128", nvec=1, nmax=10, dt=0.01),
        # S^zz(q, w) of the 24-site chain at all 13 wave numbers, 200 frequencies
        dict(name="spectrum_chain24_f32", path="spectrum", model="spin", lattice="chain", lx=24, ly=1, n_up=12,
             n_dn=0, random_j=False, dtype="f32", nq=13, nz=200, steps=48),
        # the batched solver: chains of mixed length, each with its own couplings
        dict(name="batch_chains_f64", path="batch", model="spin", lattice="chain", lx=16, ly=1, n_up=8, n_dn=0,
             random_j=True, dtype="f64", n_min=12, nprob=200, tol=1e-12, check_every=8),
    ]


def draw(rng):
    path = rng.choice(["apply", "apply", "apply", "lanczos", "ground", "reorth", "tpq", "evolve", "spectrum",
                       "batch"])
    rj = rng.random() < 0.5
    if path in ("apply", "lanczos") and rng.random() < 0.65:
        # spin sector: lengths of the configured chains, ladders and square lattices, off-centre sectors too
        kind = rng.choice(["chain", "square", "square"])
        if kind == "chain":
            lx, ly = rng.randint(*((12, 29) if path == "apply" else (16, 28))), 1
        else:
            ly = rng.choice([2, 2, 3, 4, 5])
            lx = rng.randint(max(3, 13 // ly + 1), (30 if path == "apply" else 28) // ly)
        n = lx * ly
        n_up = n // 2 - rng.choice([0, 0, 1, 2])
        c = dict(path=path, model="spin", lattice=kind, lx=lx, ly=ly, n_up=n_up, n_dn=0, random_j=rj,
                 dtype=rng.choice(["f32", "f64"]))
        if path == "lanczos":
            return dict(c, steps=rng.randint(8, 20))
        nvec = rng.choice([1, 1, 1, 1, 2, rng.randint(3, 16)]) if n <= 24 else 1
        if nvec > 1 and rng.random() < 0.5:
            c["dtype"] = rng.choice(["c64", "c128"])
        return dict(c, nvec=nvec, beta=rng.choice([0.0, 0.0, 0.5]))
    if path in ("apply", "lanczos", "reorth", "evolve"):
        lx, ly = rng.choice([(8, 1), (9, 1), (10, 1), (11, 1), (4, 2), (5, 2), (6, 2), (7, 2), (13, 1)])
        if path == "apply" and rng.random() < 0.15:
            lx, ly = 4, 4
        n = lx * ly
        n_up, n_dn = n // 2, n // 2 - rng.choice([0, 0, 1])
        c = dict(path=path, model="hubbard", lattice="square" if ly > 1 else "chain", lx=lx, ly=ly, n_up=n_up,
                 n_dn=n_dn, random_j=rj)
        if path == "apply":
            return dict(c, dtype=rng.choice(["f32", "f64"] if n == 16 else ["f32", "f64", "c128"]),
                        nvec=1 if n == 16 else rng.choice([1, 1, 1, 2, 5]), beta=rng.choice([0.0, 0.5]))
        if path == "evolve":
            return dict(c, dtype=rng.choice(["c64", "c128"]), nvec=rng.choice([1, 1, 2, 3]), nmax=rng.choice([4, 10]),
                        dt=0.01)
        return dict(c, dtype=rng.choice(["f32", "f64"]), steps=rng.randint(12, 40) if path == "reorth" else 16)
    if path == "ground":
        n = rng.randint(14, 22)
        return dict(path=path, model="spin", lattice="chain", lx=n, ly=1, n_up=n // 2, n_dn=0, random_j=rj,
                    dtype="f64", tol=1e-12, check_every=rng.choice([1, 4, 8]))
    if path == "tpq":
        kind = rng.choice(["chain", "rrg"])
        dtype = rng.choice(["c64", "c128"])
        most = 25 if dtype == "c64" else 22
        n = 2 * rng.randint(7, most // 2) if kind == "rrg" else rng.randint(13, most)
        return dict(path=path, model="full", lattice=kind, lx=n, ly=1, n_up=0, n_dn=0, random_j=True,
                    dtype=dtype, nvec=rng.choice([16, 16, 16, 1, rng.randint(2, 15)]),
                    nmax=rng.choice([1, 6, 6]), dtau=0.02)
    if path == "spectrum":
        n = rng.randint(15, 23)
        return dict(path=path, model="spin", lattice="chain", lx=n, ly=1, n_up=n // 2, n_dn=0, random_j=False,
                    dtype=rng.choice(["f32", "f64"]), nq=rng.randint(1, 16), nz=rng.randint(50, 200),
                    steps=rng.randint(16, 48))
    n = rng.randint(13, 16)
    return dict(path="batch", model="spin", lattice="chain", lx=n, ly=1, n_up=n // 2, n_dn=0, random_j=True,
                dtype="f64", n_min=rng.randint(10, n), nprob=rng.randint(20, 200), tol=1e-12,
                check_every=rng.choice([4, 8]))


# ---- inputs ------------------------------------------------------------------

def _sites(case):
    return case["lx"] * case["ly"]


def _bonds(case):
    kind, lx, ly = case["lattice"], case["lx"], case["ly"]
    if kind == "rrg":  # 3-regular graph, the same for every seed: pairing with rejection
        rng = random.Random(lx)
        while True:
            stubs = [v for v in range(lx) for _ in range(3)]
            rng.shuffle(stubs)
            edges = {(min(a, b), max(a, b)) for a, b in zip(stubs[0::2], stubs[1::2])}
            if len(edges) == 3 * lx // 2 and all(a != b for a, b in edges):
                return sorted(edges)
    if kind == "ladder":  # two legs and one extra site at the end: an odd number of sites
        e = [(i, i + 2) for i in range(2 * lx - 2)] + [(2 * i, 2 * i + 1) for i in range(lx)]
        return e + [(2 * lx - 1, 2 * lx), (0, 2 * lx)]
    e = set()
    for y in range(ly):
        for x in range(lx):
            s = x + lx * y
            for t in ((x + 1) % lx + lx * y, x + lx * ((y + 1) % ly)):
                if s != t:
                    e.add((min(s, t), max(s, t)))
    return sorted(e)


def _n(case):
    return _sites(case) + (1 if case["lattice"] == "ladder" else 0)


def _couplings(case, n, seed):
    if not case["random_j"]:
        return [1.0] * n
    r = random.Random(1000 + seed)
    return [r.uniform(0.5, 1.5) for _ in range(n)]


def _terms(case, seed):
    b = _bonds(case)
    js = _couplings(case, len(b), seed)
    if case["model"] == "hubbard":
        return [("HOP", i, j, -1, t, 0.0) for (i, j), t in zip(b, js)] + [
            ("HUBBARD_U", i, i, 0, 8.0, 0.0) for i in range(_n(case))]
    return [("EXCHANGE", i, j, 0, j_, 0.0) for (i, j), j_ in zip(b, js)]


def _dim(case):
    n = _n(case)
    if case["model"] == "full":
        return 1 << n
    if case["model"] == "hubbard":
        return math.comb(n, case["n_up"]) * math.comb(n, case["n_dn"])
    return math.comb(n, case["n_up"])


def _randn(shape, dtype, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.randn(shape, dtype=dtype, device="cuda", generator=g)


def _normalised(shape, dtype, seed):
    v = _randn(shape, dtype, seed)
    real = torch.view_as_real(v) if v.is_complex() else v.unsqueeze(-1)
    norm2 = sum(part.double().square().sum(dim=(0, -1)) for part in real.split(1 << 22))  # a slab at a time
    return v.div_(norm2.sqrt().to(real.dtype))


def _block(case, seed):
    """The vector or block of columns that the pass starts from."""
    d, dt = _dim(case), DTYPES[case["dtype"]]
    nvec = case.get("nvec", 1)
    shape = (d,) if nvec == 1 else (d, nvec)
    if case["path"] == "apply":
        return _randn(shape, dt, seed)
    return _normalised(shape, dt, seed)


def _batch_sizes(case):
    n, lo = case["lx"], case["n_min"]
    return [lo + p % (n - lo + 1) for p in range(case["nprob"])]


def _batch_case(case, n):
    return dict(case, path="ground", lx=n, n_up=n // 2)


def _shifts(case, seed):
    r = np.random.RandomState(seed % (1 << 31))
    q = 2.0 * np.pi * np.arange(case["nq"]) / case["lx"]
    e = -0.44 * case["lx"]
    return q, e + np.sort(r.uniform(0.0, 4.0, case["nz"])) + 0.05j


@functools.lru_cache(maxsize=None)
def _ctx():
    return hphi.Context(0)  # one context for the life of the program


def _ham(case, seed):
    model = {"spin": "SPIN_HALF", "full": "SPIN_HALF_GC", "hubbard": "HUBBARD"}[case["model"]]
    basis = hphi.Basis(_ctx(), model, _n(case), case["n_up"], case["n_dn"])
    return hphi.Hamiltonian(_ctx(), basis, _terms(case, seed))


def prepare(case, seed):
    s = dict(case=case)
    path = case["path"]
    if path == "batch":
        cs = [_batch_case(case, n) for n in _batch_sizes(case)]
        s["hams"] = [_ham(c, seed + p) for p, c in enumerate(cs)]
        s["v0s"] = [_block(c, seed + p) for p, c in enumerate(cs)]
        s["gs"] = torch.zeros(sum(v.numel() for v in s["v0s"]), dtype=torch.float64, device="cuda")
        s["gss"] = list(s["gs"].split([v.numel() for v in s["v0s"]]))
        return s
    s["ham"] = _ham(case, seed)
    x = _block(case, seed)
    s["x"] = x
    if path == "apply":
        s["y"] = _randn(tuple(x.shape), x.dtype, seed + 1) if case["beta"] else torch.empty_like(x)
    elif path in ("ground", "reorth"):
        s["gs"] = torch.empty_like(x)
    elif path == "tpq":
        s["norm2"] = np.ones(case["nvec"])
    elif path == "spectrum":
        s["q"], s["z"] = _shifts(case, seed)
    return s


# ---- one pass ------------------------------------------------------------------

def _scalars(case, *arrays):
    """Host scalars in the precision of the vectors they were reduced from."""
    t = {"f32": np.float32, "c64": np.float32}.get(case["dtype"], np.float64)
    c = {"f32": np.complex64, "c64": np.complex64}.get(case["dtype"], np.complex128)
    return [np.asarray(a).astype(c if np.iscomplexobj(a) else t) for a in arrays]


def run(state):
    case = state["case"]
    path = case["path"]
    if path == "batch":
        r = hphi.hphi_lanczos_batch(state["hams"], state["v0s"], 300, case["tol"], case["check_every"], state["gss"])
        return {"e0": np.array([p["e0"] for p in r]), "gs": state["gs"]}
    ham, x = state["ham"], state["x"]
    if path == "apply":
        return hphi.hphi_apply_H(ham, x, state["y"], 1.0, case["beta"])
    if path == "lanczos":
        r = hphi.hphi_lanczos(ham, x, case["steps"], 0.0, case["steps"])
        return _scalars(case, r["alpha"], r["beta"], [r["e0"]])
    if path == "ground":
        r = hphi.hphi_lanczos(ham, x, 300, case["tol"], case["check_every"], state["gs"])
        return {"e0": r["e0"], "gs": state["gs"]}
    if path == "reorth":
        r = hphi.hphi_lanczos(ham, x, case["steps"], 0.0, case["steps"], state["gs"], True)
        return _scalars(case, r["alpha"], r["beta"], [r["e0"]]) + [state["gs"]]
    if path == "tpq":
        e, h2, logd = hphi.hphi_tpq_step(ham, x, case["dtau"], case["nmax"], state["norm2"])
        return [x] + _scalars(case, e, h2, logd, state["norm2"])
    if path == "evolve":
        return [x] + _scalars(case, *hphi.hphi_time_step(ham, x, case["dt"], case["nmax"]))
    _, d, info = hphi.hphi_szz_spectrum(ham, x, state["q"], state["z"], case["steps"], 0.0, case["steps"])
    return _scalars(case, d, info["resid"])


# ---- what a pass cannot do without ---------------------------------------------

def _apply_work(case, d, cols, size, vectors):
    """Bytes and operations of one product of `cols` real columns that moves `vectors` vectors."""
    n, nb = _n(case), len(_bonds(case))
    if case["model"] == "hubbard":
        hops = sum(2.0 * k * (n - k) / (n * (n - 1)) for k in (case["n_up"], case["n_dn"])) * nb
    elif case["model"] == "full":
        hops = 0.5 * nb
    else:
        hops = 2.0 * case["n_up"] * (n - case["n_up"]) / (n * (n - 1)) * nb
    return float(vectors) * d * cols * size, 2.0 * (hops + 1.0) * d * cols


def work(case):
    path = case["path"]
    if path == "batch":
        b = f = 0.0
        for n in _batch_sizes(case):
            c = _batch_case(case, n)
            d = _dim(c)
            _, f1 = _apply_work(c, d, 1, 8, 2)
            b += 2.0 * d * 8
            f += 2 * 50 * (f1 + 8.0 * d)
        return {"bytes": b, "flops": f}
    d = _dim(case)
    size = 4 if case["dtype"] in ("f32", "c64") else 8
    cols = case.get("nvec", 1) * (2 if case["dtype"].startswith("c") else 1)
    if path == "apply":
        b, f = _apply_work(case, d, cols, size, 3 if case["beta"] else 2)
    elif path in ("tpq", "evolve"):  # each stage reads V and W and writes W
        b, f = _apply_work(case, d, cols, size, 3)
        b, f = b * case["nmax"], f * case["nmax"]
    elif path == "spectrum":
        cols = 2 * case["nq"]
        b, f = _apply_work(case, d, cols, size, 3 + 3)
        b, f = b * case["steps"], (f + 8.0 * d * cols) * case["steps"]
    else:
        steps = case.get("steps", 60)
        b, f = _apply_work(case, d, 1, size, 3 + 3)
        b, f = b * steps, (f + 8.0 * d) * steps
        if path == "ground":
            b, f = 2 * b, 2 * f
        if path == "reorth":  # two projection passes over the vectors kept so far
            b += 4.0 * d * size * steps * (steps + 1) / 2
            f += 8.0 * d * steps * (steps + 1) / 2
    return {"bytes": b, "flops": f}


# ---- the same in 64 bits, without the library ------------------------------------

def _states(n, k):
    """Ascending n-bit strings with k bits set, and the inverse tables (rank = hi[s >> lo] + low[s & mask])."""
    lo = n - n // 2
    s = torch.arange(1 << lo, device="cuda")
    pop = sum((s >> b) & 1 for b in range(lo))
    low = torch.empty_like(s)
    classes = []
    for p in range(lo + 1):
        c = (pop == p).nonzero().flatten()
        low[c] = torch.arange(c.numel(), device="cuda")
        classes.append(c)
    h = torch.arange(1 << (n // 2), device="cuda")
    need = k - sum((h >> b) & 1 for b in range(n // 2))
    count = torch.tensor([c.numel() for c in classes], device="cuda")
    length = torch.where((need >= 0) & (need <= lo), count[need.clamp(0, lo)], torch.zeros_like(need))
    hi = length.cumsum(0) - length
    first = count.cumsum(0) - count
    at = torch.repeat_interleave(first[need.clamp(0, lo)] - hi, length) + torch.arange(int(length.sum()), device="cuda")
    states = torch.cat(classes)[at] | (torch.repeat_interleave(h, length) << lo)
    return states, lambda t: hi[t >> lo] + low[t & ((1 << lo) - 1)]


class _Exact:
    """H of a case in 64 bits, acting on [D] or [D][columns]."""

    def __init__(self, case, seed):
        self.case, self.n = case, _n(case)
        self.bonds = _bonds(case)
        self.js = _couplings(case, len(self.bonds), seed)
        if case["model"] == "hubbard":
            self.species = [self._hops(case["n_up"]), self._hops(case["n_dn"])]
            up, dn = self.species[0][0], self.species[1][0]
            self.diag = torch.zeros((up.numel(), dn.numel()), dtype=torch.float64, device="cuda")
            for i in range(self.n):
                self.diag += 8.0 * ((up >> i) & 1)[:, None] * ((dn >> i) & 1)[None, :]
        elif case["model"] == "full":
            s = torch.arange(1 << self.n, device="cuda")
            self.diag = sum(0.25 * j * (1 - 2 * (((s >> a) ^ (s >> b)) & 1)).double()
                            for (a, b), j in zip(self.bonds, self.js))
        else:
            self.states, self.rank = _states(self.n, case["n_up"])
            self.small = None
            if self.states.numel() <= 20_000:  # all targets at once: [bonds][D]
                m = torch.tensor([(1 << i) | (1 << j) for i, j in self.bonds], device="cuda")[:, None]
                t = self.states & m
                self.small = self.rank(torch.where((t != 0) & (t != m), self.states ^ m, self.states))
                self.j = torch.tensor(self.js, dtype=torch.float64, device="cuda")

    def _hops(self, k):
        s, rank = _states(self.n, k)
        out = []
        for (i, j), t in zip(self.bonds, self.js):
            rows = ((((s >> i) ^ (s >> j)) & 1) == 1).nonzero().flatten()
            between = s[rows] & (((1 << j) - 1) & ~((2 << i) - 1))
            odd = sum((between >> b) & 1 for b in range(self.n)) & 1
            out.append((rows, rank(s[rows] ^ ((1 << i) | (1 << j))), (-t) * (1 - 2 * odd).double()))
        return s, out

    def __call__(self, x):
        if self.case["model"] == "hubbard":
            shape = (self.species[0][0].numel(), self.species[1][0].numel()) + tuple(x.shape[1:])
            xs = x.reshape(shape)
            y = self.diag.reshape(shape[:2] + (1,) * (xs.dim() - 2)) * xs
            for dim in (0, 1):
                for rows, target, c in self.species[dim][1]:
                    c = c.reshape((-1,) + (1,) * (xs.dim() - 1 - dim))
                    y.index_add_(dim, rows, c * xs.index_select(dim, target))
            return y.reshape(x.shape)
        if self.case["model"] == "full":
            y = x * self.diag.reshape((-1,) + (1,) * (x.dim() - 1))
            for (i, j), v in zip(self.bonds, self.js):
                view = (1 << (self.n - 1 - j), 2, 1 << (j - i - 1), 2, -1)
                xv, yv = x.view(view), y.view(view)
                yv[:, 0, :, 1].add_(xv[:, 1, :, 0], alpha=0.5 * v)
                yv[:, 1, :, 0].add_(xv[:, 0, :, 1], alpha=0.5 * v)
            return y
        if self.small is not None and x.dim() == 1:
            return 0.5 * (self.j @ x[self.small]) - 0.25 * self.j.sum() * x
        y = torch.empty_like(x)
        chunk = max(1 << 16, (1 << 26) // max(1, x[:1].numel()))
        for a in range(0, x.shape[0], chunk):
            s = self.states[a:a + chunk]
            xa = x[a:a + chunk]
            acc = torch.zeros_like(xa)
            for (i, j), v in zip(self.bonds, self.js):
                differ = ((s >> i) ^ (s >> j)) & 1
                off = x[self.rank(s ^ (differ * ((1 << i) | (1 << j))))]  # the row itself where the spins agree
                acc.add_(off, alpha=0.5 * v).sub_(xa, alpha=0.25 * v)
            y[a:a + chunk] = acc
        return y


def _krylov(h, v0, steps, tol=None):
    """Reorthogonalised Lanczos: (alpha, beta[1..], basis vectors, Ritz values, Ritz vectors)."""
    vs = torch.empty((steps, v0.numel()), dtype=torch.float64, device="cuda")
    vs[0] = v0 / v0.norm()
    alpha, beta = [], []
    while True:
        m = len(alpha) + 1
        u = h(vs[m - 1])
        alpha.append(float(torch.dot(vs[m - 1], u)))
        for _ in range(2):
            u -= (vs[:m] @ u) @ vs[:m]
        beta.append(float(u.norm()))
        if m == steps or (tol and m % 8 == 0) or beta[-1] < 1e-13:
            t = np.diag(alpha) + np.diag(beta[:m - 1], 1) + np.diag(beta[:m - 1], -1)
            w, y = np.linalg.eigh(t)
            if m == steps or beta[-1] < 1e-13 or (tol and beta[-1] * abs(y[-1, 0]) < tol):
                return np.array(alpha), np.array(beta), vs, w, y
        vs[m] = u / beta[-1]


def _ritz(vs, y):
    y = y[:, 0] * (1.0 if y[0, 0] >= 0 else -1.0)
    g = torch.from_numpy(y.copy()).to(vs.device) @ vs[:len(y)]
    return g / g.norm()


def _ground(case, seed):
    _, _, vs, w, y = _krylov(_Exact(case, seed), _block(case, seed).double(), 280, 1e-13)
    return float(w[0]), _ritz(vs, y)


def exact(case, seed):
    path = case["path"]
    if path == "batch":
        got = [_ground(_batch_case(case, n), seed + p) for p, n in enumerate(_batch_sizes(case))]
        return {"e0": np.array([e for e, _ in got]), "gs": torch.cat([g for _, g in got])}
    if path == "ground":
        e0, gs = _ground(case, seed)
        return {"e0": e0, "gs": gs}
    if path == "lanczos" and _dim(case) > 50_000_000:
        return None  # the reorthogonalised run would take too long
    h = _Exact(case, seed)
    x = _block(case, seed)
    x = x.to(torch.complex128 if x.is_complex() else torch.float64)
    if path == "apply":
        y = h(x)
        if case["beta"]:
            y += case["beta"] * _randn(tuple(x.shape), DTYPES[case["dtype"]], seed + 1)
        return y
    if path in ("lanczos", "reorth"):
        alpha, beta, vs, w, y = _krylov(h, x, case["steps"])
        return [alpha, beta, np.array(w[:1])] + ([_ritz(vs, y)] if path == "reorth" else [])
    if path in ("tpq", "evolve"):
        v = x.reshape(x.shape[0], -1)
        hv = h(v)
        n2 = v.abs().square().sum(0)
        e = (v.conj() * hv).sum(0).real / n2
        h2 = hv.abs().square().sum(0) / n2
        del hv
        c = -0.5 * case["dtau"] if path == "tpq" else -1j * case["dt"]
        w = v  # the Taylor sum in Horner form
        for k in range(case["nmax"], 0, -1):
            w = h(w).mul_(c / k).add_(v)
        new = w.abs().square().sum(0)
        n2, e, h2, new = (t.cpu().numpy() for t in (n2, e, h2, new))
        if path == "evolve":
            return [w.reshape(x.shape), n2, e, h2, new]
        # the library takes norm2 = 1 as given and returns V / |V| evolved
        return [w.reshape(x.shape), e, h2, np.log(new / n2), new]
    # spectrum: continued fraction of each real column's own Krylov space
    q, z = _shifts(case, seed)
    n = _n(case)
    d, resid = np.zeros((q.size, z.size), complex), np.zeros((q.size, z.size))
    if q.size * _dim(case) > 40_000_000:
        return None  # over the time that a check may take
    for a, qa in enumerate(q):
        spin = sum(np.exp(1j * qa * l) * (((h.states >> l) & 1).double() - 0.5) for l in range(n))
        worst = np.zeros(z.size)
        for b in (spin.real * x, spin.imag * x):
            if float(b.norm()) < 1e-13:
                continue
            alpha, beta, _, _, _ = _krylov(h, b, case["steps"])
            m = len(alpha)
            f = z - alpha[m - 1]
            for k in range(m - 2, -1, -1):
                f = z - alpha[k] - beta[k] ** 2 / f
            d[a] += float(b.square().sum()) / f
            u = rho = None
            for k in range(m):
                u = z - alpha[k] - (beta[k - 1] ** 2 / u if k else 0.0)
                rho = beta[k] / np.abs(u) * (rho if k else 1.0)
            worst = np.maximum(worst, rho)
        resid[a] = worst
    return [d, resid]
