"""Timed cases of the library: the calls a user's program makes, over the sizes it makes them at.

A case is a dict of plain values; its "kind" names the public call:

  matvec        y = H x of one sector (api.matvec), one vector or a block of them
  lanczos       a whole Lanczos run from a given start vector (api.lanczos_run)
  autograd      y = H(J) x and its backward pass (autograd.HeisenbergMatvec)
  ground_state  E0 and dE0/dJ (api.e0_grad)
  ftlm          a finite-temperature run over all sectors (api.ftlm_run)
  arnoldi       an Arnoldi run with full re-orthogonalisation (api.arnoldi_run)

"lattice" names the bonds: "ring" (J1 = -1), "j1j2" (J1 = -1 and "j2"), "randj" (the bonds of
"j1j2" with couplings uniform in [-1.2, -0.8]) or "graph" (each site bonded to 4 random partners,
couplings uniform in [-1.5, -0.5]).  The sector is (n, two_s, two_m), or its momentum-0 block
when "momentum" is set.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_0706_3293_gb300 import api, workloads
from paper_0706_3293_gb300.autograd import HeisenbergMatvec

_DTYPE = {"f64": torch.float64, "f32": torch.float32}


def listed():
    return [
        # a whole run on a small sector, 12,870 rows: launches and latency are what it costs
        dict(name="lanczos_ring16_f64", kind="lanczos", n=16, two_s=1, two_m=0, lattice="ring", dtype="f64", steps=40),
        # one product of a mid-size frustrated ring, 184,756 rows, as iterative solvers of the
        # caller's own (time evolution, kernel polynomials) ask for it thousands of times
        dict(name="matvec_j1j2_20_f64", kind="matvec", n=20, two_s=1, two_m=0, lattice="j1j2", j2=-0.5, dtype="f64",
             nvec=1),
        # the same for a block of vectors at once (random-phase traces, block methods)
        dict(name="matvec_block8_j1j2_20_f64", kind="matvec", n=20, two_s=1, two_m=0, lattice="j1j2", j2=-0.3,
             dtype="f64", nvec=8),
        # a higher spin: the rings of spins s = 3/2 of magnetic molecules, 1.7 M rows
        dict(name="matvec_s32_ring12_f64", kind="matvec", n=12, two_s=3, two_m=0, lattice="ring", dtype="f64", nvec=1),
        # a symmetry block: momentum 0 of the 28-site ring, 1.4 M representatives of 40 M states
        dict(name="matvec_k0_j1j2_28_f64", kind="matvec", n=28, two_s=1, two_m=0, lattice="j1j2", j2=-0.5, dtype="f64",
             nvec=1, momentum=True),
        # single-precision vectors on an odd ring (ragged blocks, M = 1/2), 20 M rows
        dict(name="lanczos_ring27_f32", kind="lanczos", n=27, two_s=1, two_m=1, lattice="ring", dtype="f32", steps=12),
        # s = 1 on a random graph, single precision, 44 M rows
        dict(name="lanczos_s1_graph18_f32", kind="lanczos", n=18, two_s=2, two_m=0, lattice="graph", dtype="f32",
             steps=12),
        # the largest sector: 601 M rows, the first steps of a ground-state run
        dict(name="lanczos_j1j2_32_f64", kind="lanczos", n=32, two_s=1, two_m=0, lattice="j1j2", j2=-0.5, dtype="f64",
             steps=8),
        # a training step of fitted couplings: product, dL/dx and dL/dJ for 48 couplings, 2.7 M rows
        dict(name="autograd_randj_24_f64", kind="autograd", n=24, two_s=1, two_m=0, lattice="randj", dtype="f64"),
        # the ground-state gradient with respect to 36 couplings, 48,620 rows
        dict(name="ground_state_randj_18", kind="ground_state", n=18, two_s=1, two_m=0, lattice="randj", steps=120),
        # thermodynamics of a ring from 32 random vectors in each of its 21 sectors
        dict(name="ftlm_j1j2_20", kind="ftlm", n=20, lattice="j1j2", j2=-0.3, R=32, steps=80),
        # Krylov space with full re-orthogonalisation, 705,432 rows
        dict(name="arnoldi_j1j2_22", kind="arnoldi", n=22, two_s=1, two_m=0, lattice="j1j2", j2=-0.3, steps=40),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["matvec", "matvec", "matvec", "lanczos", "lanczos", "autograd", "ground_state", "ftlm",
                       "arnoldi"])
    j2 = rng.choice([-0.2, -0.25, -0.3, -0.5, -0.6])
    if kind == "ftlm":
        return dict(kind=kind, n=rng.randint(10, 20), lattice="j1j2", j2=j2, R=rng.randint(1, 32),
                    steps=rng.randint(40, 90))
    if kind in ("autograd", "ground_state"):
        n = rng.randint(12, 24) if kind == "autograd" else rng.randint(10, 18)
        case = dict(kind=kind, n=n, two_s=1, two_m=n % 2 + 2 * rng.choice([0, 0, 1]), lattice="randj")
        case.update({"dtype": rng.choice(["f64", "f64", "f32"])} if kind == "autograd" else {"steps": rng.randint(90, 150)})
        return case
    # the sector: its spin, then a number of rows spread over the range, then the largest n
    # whose sector has no more rows
    two_s = rng.choice([1, 1, 1, 1, 2, 2, 3, 4, 5])
    top = {1: 4e7, 2: 4.5e7}.get(two_s, 2.5e6)
    if kind == "arnoldi":
        top = 1.5e6
    rows = _log_uniform(rng, 300, top)
    extra = rng.choice([0, 0, 2, 4])            # 2M above its smallest value
    n = 4
    while _dim(n + 1, two_s, ((n + 1) * two_s) % 2 + extra) <= rows:
        n += 1
    lattice = rng.choice(["ring", "j1j2", "j1j2", "randj", "graph"]) if n >= 6 else "ring"
    case = dict(kind=kind, n=n, two_s=two_s, two_m=(n * two_s) % 2 + extra, lattice=lattice,
                dtype="f64" if kind == "arnoldi" else rng.choice(["f64", "f32"]))
    if lattice == "j1j2":
        case["j2"] = j2
    if kind == "matvec":
        case["nvec"] = rng.choice([1, 1, 1, 2, 3, 4, 7, 8, 16, 33]) if _dim_of(case) <= 2.5e6 else 1
        if lattice in ("ring", "j1j2") and case["nvec"] == 1 and rng.random() < 0.3:
            case["momentum"] = True
    else:
        # short enough that no Ritz value converges to the vectors' precision, after which the
        # recurrence of plain Lanczos is no longer determined by its start vector
        dim = _dim_of(case)
        case["steps"] = min(rng.randint(8, 14) if case["dtype"] == "f32" else rng.randint(12, 32), max(4, dim // 40))
    return case


# ---- inputs ---------------------------------------------------------------------------------

def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) & (2**62 - 1))


def _uniform(shape, dtype, gen):
    return torch.rand(shape, dtype=dtype, device="cuda", generator=gen).mul_(2).sub_(1)


def _bonds(case, seed):
    """(u, v, J) host arrays; couplings drawn at random come from the seed, the graph from n."""
    n, kind = case["n"], case["lattice"]
    if kind == "graph":
        u, v = workloads.random_regular_graph(n, 4, 3)
        return u, v, workloads.uniform_couplings(len(u), -1.5, -0.5, int(seed) & (2**62 - 1))
    u, v, J = workloads.ring_bonds(n, -1.0, None if kind == "ring" else case.get("j2", -1.0))
    if kind == "randj":
        J = workloads.uniform_couplings(len(u), -1.2, -0.8, int(seed) & (2**62 - 1))
    return u, v, J


def _temperatures():
    return np.geomspace(0.1, 10.0, 24)


def prepare(case, seed):
    u, v, J = _bonds(case, seed)
    state = dict(case=case, bonds=api.BondList.make(u, v, J), seed=int(seed) & (2**62 - 1))
    if case["kind"] == "ftlm":
        return state
    basis = api.Basis(case["n"], case["two_s"], case["two_m"], momentum=0 if case.get("momentum") else None)
    state["basis"] = basis
    gen = _generator(seed)
    dtype = _DTYPE[case.get("dtype", "f64")]
    nvec = case.get("nvec", 1)
    state["x"] = _uniform(basis.dim if nvec == 1 else (basis.dim, nvec), dtype, gen)
    if case["kind"] == "autograd":
        state["x"].requires_grad_()
        state["J"] = torch.from_numpy(J).requires_grad_()
        state["g"] = torch.randn(basis.dim, dtype=dtype, device="cuda", generator=gen)
    return state


def run(state):
    case, bonds = state["case"], state["bonds"]
    kind = case["kind"]
    if kind == "ftlm":
        r = api.ftlm_run(case["n"], bonds, case["R"], case["steps"], state["seed"], _temperatures())
        return {"Z": r.Z, "E": r.E, "e_ref": r.e_ref}
    basis, x = state["basis"], state["x"]
    if kind == "matvec":
        return api.matvec(basis, bonds, x)
    if kind == "lanczos":
        r = api.lanczos_run(basis, bonds, case["steps"], v0=x, dtype=x.dtype, n_ritz=3)
        return {"alpha": r.alpha, "beta": r.beta, "ritz": r.ritz}
    if kind == "autograd":
        y = HeisenbergMatvec.apply(x, state["J"], basis, bonds.u, bonds.v)
        gx, gJ = torch.autograd.grad(y, (x, state["J"]), state["g"])
        return {"y": y.detach(), "grad_x": gx, "grad_J": gJ}
    if kind == "ground_state":
        e0, grad, _, _ = api.e0_grad(basis, bonds, case["steps"], v0=x)
        return {"e0": e0, "grad_J": grad}
    r = api.arnoldi_run(basis, bonds, case["steps"], v0=x, n_ritz=3)
    return {"H": r.H, "ritz": r.ritz}


# ---- counts ---------------------------------------------------------------------------------

def _counts(n, two_s):
    """Number of n-site states of each digit sum."""
    c = [1]
    for _ in range(n):
        d = [0] * (len(c) + two_s)
        for a, k in enumerate(c):
            for t in range(two_s + 1):
                d[a + t] += k
        c = d
    return c


def _dim(n, two_s, two_m):
    c = _counts(n, two_s)
    a = (n * two_s - two_m) // 2
    return c[a] if 0 <= a < len(c) else 0


def _dim_of(case):
    return _dim(case["n"], case["two_s"], case["two_m"])


def _n_bonds(case):
    return case["n"] * {"ring": 1, "j1j2": 2, "randj": 2, "graph": 2}[case["lattice"]]


def _nnz(n, two_s, a, n_bonds):
    """Matrix elements of one sector: its diagonal and both exchanges of every bond."""
    c, rest = _counts(n, two_s), _counts(n - 2, two_s)
    hops = sum(rest[a - p - q] for p in range(1, two_s + 1) for q in range(two_s) if 0 <= a - p - q < len(rest))
    return c[a] + 2 * n_bonds * hops


def work(case):
    kind, n = case["kind"], case["n"]
    nb = _n_bonds(case)
    if kind == "ftlm":
        rows = 2 ** n
        nnz = sum(_nnz(n, 1, a, nb) for a in range(n + 1))
        vec = case["R"] * case["steps"]
        return {"bytes": 12 * rows * vec, "flops": (2 * nnz + 8 * rows) * vec}
    two_s = case["two_s"]
    dim = _dim_of(case)
    nnz = _nnz(n, two_s, (n * two_s - case["two_m"]) // 2, nb)
    if case.get("momentum"):
        dim, nnz = -(-dim // n), -(-nnz // n)      # orbits of full period, up to the few shorter ones
    es = 4 if case.get("dtype") == "f32" else 8
    if kind == "matvec":
        nvec = case["nvec"]
        return {"bytes": 2 * dim * es * nvec, "flops": 2 * nnz * nvec}
    if kind == "autograd":                         # x, g in; y, grad_x out; three products
        return {"bytes": 4 * dim * es, "flops": 6 * nnz}
    steps = case["steps"]
    if kind == "arnoldi":                          # step j: product, two Gram-Schmidt passes over j vectors
        pairs = steps * (steps + 1) // 2
        return {"bytes": dim * es * (3 * steps + 2 * pairs), "flops": 2 * nnz * steps + 8 * dim * pairs}
    passes = 2 if kind == "ground_state" else 1    # the second one accumulates the eigenvector
    return {"bytes": dim * es * (1 + 3 * steps * passes), "flops": (2 * nnz + 8 * dim) * steps * passes}


# ---- the same results in 64 bits, in plain torch ---------------------------------------------------

class _Sector:
    """H on one sector: its states as packed digits in index order, a product in float64."""

    def __init__(self, n, two_s, a, bonds, momentum=False):
        self.two_s, self.bits = two_s, 1 if two_s == 1 else 2 if two_s <= 3 else 4
        b = self.bits
        sums = {0: torch.zeros(1, dtype=torch.int64, device="cuda")}
        for p in range(n):
            nxt = {}
            for s in range(a + 1):
                parts = [sums[s - d] | (d << (b * p)) for d in range(two_s + 1) if s - d in sums]
                if parts and s + two_s * (n - 1 - p) >= a:
                    nxt[s] = torch.cat(parts)
            sums = nxt
        self.states, self.period = sums[a], None
        if momentum:
            full, w = (1 << (b * n)) - 1, self.states
            rep, period = w.clone(), torch.full_like(w, n)
            for k in range(1, n):
                t = ((w << (b * k)) | (w >> (b * (n - k)))) & full
                period = torch.where((t == w) & (period == n), torch.full_like(w, k), period)
                rep = torch.minimum(rep, t)
            keep = rep == w
            self.states, self.period, self.n = w[keep], period[keep], n
        self.dim = self.states.numel()
        self.bonds = [(int(min(p, q)), int(max(p, q)), float(j)) for p, q, j in zip(*bonds)]
        self.kept = {} if self.dim * len(self.bonds) * 40 <= 70e9 else None

    def _digit(self, p):
        return (self.states >> (self.bits * p)) & ((1 << self.bits) - 1)

    def _target(self, p, q, d):
        w = self.states + d * ((1 << (self.bits * p)) - (1 << (self.bits * q)))
        if self.period is not None:
            full, b, n = (1 << (self.bits * self.n)) - 1, self.bits, self.n
            rep = w.clone()
            for k in range(1, n):
                rep = torch.minimum(rep, ((w << (b * k)) | (w >> (b * (n - k)))) & full)
            w = rep
        return torch.searchsorted(self.states, w).clamp_(max=self.dim - 1)

    def _terms(self, b):
        """s_u.s_v of bond b: its diagonal and, for each exchange, factor and target of every row."""
        if self.kept is not None and b in self.kept:
            return self.kept[b]
        p, q, _ = self.bonds[b]
        s2, ap, aq = self.two_s, self._digit(p), self._digit(q)
        diag = (s2 - 2 * ap) * (s2 - 2 * aq) * 0.25
        hops = []
        for d in (-1, 1):
            if d < 0:
                f = ap * (s2 - ap + 1) * (s2 - aq) * (aq + 1)
            else:
                f = (s2 - ap) * (ap + 1) * aq * (s2 - aq + 1)
            f, t = f.double().sqrt_().mul_(0.5), self._target(p, q, d)
            if self.period is not None:
                f *= (self.period.double() / self.period[t].double()).sqrt_()
            hops.append((f, t))
        if self.kept is not None:
            self.kept[b] = (diag.double(), hops)
        return diag, hops

    def bond(self, b, x):
        """(s_u.s_v of bond b) x for x of shape [dim] or [dim, k]."""
        col = (lambda t: t) if x.dim() == 1 else (lambda t: t[:, None])
        diag, hops = self._terms(b)
        y = col(diag) * x
        for f, t in hops:
            y += col(f) * x[t]
        return y

    def apply(self, x):
        y = torch.zeros_like(x)
        for b, (_, _, j) in enumerate(self.bonds):
            y.add_(self.bond(b, x), alpha=-j)
        return y


def _sector(case, seed):
    return _Sector(case["n"], case["two_s"], (case["n"] * case["two_s"] - case["two_m"]) // 2, _bonds(case, seed),
                   bool(case.get("momentum")))


def _tridiagonal(alpha, beta):
    m = len(alpha)
    return np.diag(alpha) + np.diag(beta[: m - 1], 1) + np.diag(beta[: m - 1], -1)


def _exact_lanczos(sector, v, steps):
    v = v / v.norm()
    prev, b, alpha, beta = torch.zeros_like(v), 0.0, [], []
    for _ in range(steps):
        w = sector.apply(v) - b * prev
        a = float(torch.dot(v, w))
        w -= a * v
        b = float(w.norm())
        alpha.append(a)
        beta.append(b)
        prev, v = v, w / b
    alpha, beta = np.array(alpha), np.array(beta)
    return {"alpha": alpha, "beta": beta, "ritz": np.linalg.eigvalsh(_tridiagonal(alpha, beta))[:3]}


def _exact_krylov(sector, v, steps):
    """Arnoldi basis (rows) and Hessenberg matrix, classical Gram-Schmidt twice."""
    V = torch.zeros(steps + 1, sector.dim, dtype=torch.float64, device="cuda")
    H = np.zeros((steps + 1, steps))
    V[0] = v / v.norm()
    for j in range(steps):
        w = sector.apply(V[j])
        for _ in range(2):
            h = V[: j + 1] @ w
            w -= V[: j + 1].T @ h
            H[: j + 1, j] += h.cpu().numpy()
        beta = float(w.norm())
        H[j + 1, j] = beta
        V[j + 1] = w / beta
    return V, H


def _exact_ground_state(sector, v):
    steps = min(260, sector.dim - 1)
    V, H = _exact_krylov(sector, v, steps)
    ev, vec = np.linalg.eigh(0.5 * (H[:steps] + H[:steps].T))
    psi = V[:steps].T @ torch.from_numpy(vec[:, 0].copy()).cuda()
    psi /= psi.norm()
    grad = [-float(torch.dot(psi, sector.bond(b, psi))) for b in range(len(sector.bonds))]
    return {"e0": float(ev[0]), "grad_J": np.array(grad)}


def _splitmix(seed, t):
    """Outputs t (int64 tensor) of SplitMix64 seeded with seed (an int), as int64 bit patterns."""
    def signed(k):
        k &= 2**64 - 1
        return k - 2**64 if k >= 2**63 else k

    def shifted(z, k):                             # logical right shift
        return (z >> k) & ((1 << (64 - k)) - 1)

    z = (t + 1) * signed(0x9E3779B97F4A7C15) + signed(seed)
    z = (z ^ shifted(z, 30)) * signed(0xBF58476D1CE4E5B9)
    z = (z ^ shifted(z, 27)) * signed(0x94D049BB133111EB)
    return z ^ shifted(z, 31)


def _exact_ftlm(case, seed):
    """Thermal sums of the same random +-1 vectors, each sector by Lanczos in float64 (small
    sectors by diagonalisation)."""
    n, R, steps = case["n"], case["R"], case["steps"]
    bonds, seed = _bonds(case, seed), int(seed) & (2**62 - 1)
    theta, weight = [], []
    for a in range(n + 1):
        sector = _Sector(n, 1, a, bonds)
        D = sector.dim
        cols = []
        for r in range(R):
            key = int(_splitmix(seed, torch.tensor([a * 2**20 + r]))[0])
            o = _splitmix(key, torch.arange(D, device="cuda"))
            cols.append(torch.where(o < 0, -1.0, 1.0).double())
        v = torch.stack(cols, 1) / math.sqrt(D)
        if D <= max(2 * steps, 200):
            H = sector.apply(torch.eye(D, dtype=torch.float64, device="cuda")).cpu().numpy()
            ev, vec = np.linalg.eigh(0.5 * (H + H.T))
            tau = (vec.T @ v.cpu().numpy()) ** 2
            theta.append(np.repeat(ev, R))
            weight.append(tau.reshape(-1) * D / R)
            continue
        prev, b = torch.zeros_like(v), torch.zeros(R, dtype=torch.float64, device="cuda")
        alpha, beta = [], []
        for _ in range(steps):
            w = sector.apply(v) - b * prev
            al = (v * w).sum(0)
            w -= al * v
            b = w.norm(dim=0)
            alpha.append(al)
            beta.append(b)
            prev, v = v, w / b
        alpha, beta = torch.stack(alpha, 1).cpu().numpy(), torch.stack(beta, 1).cpu().numpy()
        for r in range(R):
            ev, vec = np.linalg.eigh(_tridiagonal(alpha[r], beta[r]))
            theta.append(ev)
            weight.append(vec[0] ** 2 * D / R)
    theta, weight = np.concatenate(theta), np.concatenate(weight)
    e_ref = float(theta.min())
    Z, E = [], []
    for T in _temperatures():
        f = weight * np.exp(-(theta - e_ref) / T)
        Z.append(f.sum())
        E.append((f * theta).sum() / f.sum())
    return {"Z": np.array(Z), "E": np.array(E), "e_ref": e_ref}


def exact(case, seed):
    kind = case["kind"]
    if kind == "ftlm":
        return _exact_ftlm(case, seed)
    if _dim_of(case) > 5e7:
        return None
    state = prepare(case, seed)
    x = state["x"].detach().double()
    sector = _sector(case, seed)
    if kind == "matvec":
        return sector.apply(x)
    if kind == "lanczos":
        return _exact_lanczos(sector, x, case["steps"])
    if kind == "autograd":
        g = state["g"].double()
        grad = [-float(torch.dot(g, sector.bond(b, x))) for b in range(len(sector.bonds))]
        return {"y": sector.apply(x), "grad_x": sector.apply(g), "grad_J": torch.tensor(grad, dtype=torch.float64)}
    if kind == "ground_state":
        return _exact_ground_state(sector, x)
    V, H = _exact_krylov(sector, x, case["steps"])
    m = case["steps"]
    return {"H": H, "ritz": np.linalg.eigvalsh(0.5 * (H[:m] + H[:m].T))[:3]}
