"""Workloads of the eigensolver as a program calls it, one pass each, for timing.

Kinds of work (the ``kind`` of a case):

* ``filter``   one rational-filter apply, ``Context.filter_apply`` -- 80 % of a solve;
* ``rr``       one outer update, ``Context.rayleigh_ritz``: B-orthogonalisation against the
               locked pairs, Cholesky-QR2, Rayleigh-Ritz, residuals;
* ``solve``    a whole ``Context.solve``;
* ``batch``    a whole ``Batch.solve`` of uneven pencils;
* ``apply``    ``Context.apply``, A X and B X;
* ``grad``     ``Context.eig_grad``, the adjoint of the eigenvalues (and of the eigenvectors).

Pencils: Q1 elements on boxes.  Scalar ones have one lognormal coefficient per element layer
of each axis (stiffness K1 x M x M + M x K1 x M + M x M x K1), the x = 0 face fixed, so that
every eigenpair is a product of one-dimensional ones and a seeded pencil comes with its exact
spectrum: interval ends, Ritz blocks and reference results need no solver.  Elasticity boxes
have a lognormal modulus per element, nu = 0.3, rho = 1 and the z = 0 face clamped.

A mixed-precision pass (``precision`` 1) solves in complex FP32, so its block and the
eigenvectors that a solve converges to a residual of 1e-8 carry single-precision digits; the
programs here keep them as FP32 tensors.  FP64 passes return what the library gives.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2510_17334_gb300 import slrf

SHIFT = 1e-3


def listed():
    return [
        # an apply late in the largest solve (64 x 64 x 32 elasticity box, Jacobi-preconditioned,
        # It_max 23): most of the wanted pairs are locked, 128 columns are still active
        {"name": "filter_elastic_large", "kind": "filter", "grid": "elastic", "nx": 64, "ny": 64, "nz": 32, "k": 128,
         "m": 8, "it": 23, "precision": 1, "warm": True, "precond": 1},
        # a warm-started apply of the scalar workload: 27 entries a row, 41^3 nodes, block 160
        {"name": "filter_scalar_mixed", "kind": "filter", "grid": "scalar", "nx": 41, "ny": 41, "nz": 41, "k": 160,
         "m": 8, "it": 8, "precision": 1, "warm": True, "precond": 0},
        # FP64 throughout, the library's default precision: odd sides, a block that fills no tile evenly
        {"name": "filter_scalar_fp64", "kind": "filter", "grid": "scalar", "nx": 31, "ny": 30, "nz": 29, "k": 75,
         "m": 8, "it": 12, "precision": 0, "warm": True, "precond": 0},
        # the smallest applies: a plane pencil, a few columns, where launches and latency count
        {"name": "filter_small_mixed", "kind": "filter", "grid": "scalar", "nx": 31, "ny": 30, "nz": 1, "k": 12,
         "m": 8, "it": 40, "precision": 1, "warm": True, "precond": 0},
        # a small apply in FP64: about as many rows and columns as the bar of the tests
        {"name": "filter_small_fp64", "kind": "filter", "grid": "scalar", "nx": 45, "ny": 44, "nz": 1, "k": 32,
         "m": 8, "it": 40, "precision": 0, "warm": True, "precond": 0},
        # the outer update between two applies of the scalar workload, some pairs locked already
        {"name": "update_scalar", "kind": "rr", "grid": "scalar", "nx": 41, "ny": 41, "nz": 41, "k": 160, "conv": 40},
        # a whole solve, mixed precision, at the default It_max: a dozen or two outer steps on a
        # block of 100
        {"name": "solve_scalar_mixed", "kind": "solve", "grid": "scalar", "nx": 21, "ny": 20, "nz": 19, "k": 100,
         "want": 66, "it": 40, "precision": 1},
        # independent uneven pencils solved together
        {"name": "batch_mixed", "kind": "batch", "count": 6, "n_lo": 2000, "n_hi": 12000, "it": 30, "precision": 1},
        # A X and B X on an elasticity box in FP64, as a program forms its own residuals
        {"name": "products_elastic", "kind": "apply", "grid": "elastic", "nx": 32, "ny": 32, "nz": 16, "k": 96,
         "fp32": False},
        # sensitivities of the lowest 50 frequencies of a 48^3 box to every stored entry
        {"name": "adjoint_values", "kind": "grad", "grid": "elastic", "nx": 48, "ny": 48, "nz": 48, "k": 50,
         "vectors": False},
        # a loss on the modes themselves: block MINRES for the eigenvector terms
        {"name": "adjoint_vectors", "kind": "grad", "grid": "scalar", "nx": 14, "ny": 13, "nz": 11, "k": 16,
         "vectors": True},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["filter", "filter", "filter", "rr", "solve", "batch", "apply", "grad", "grad"])
    if kind == "batch":
        return {"kind": "batch", "count": rng.randint(3, 6), "n_lo": 2000, "n_hi": _log_int(rng, 4000, 12000),
                "it": rng.randint(28, 36), "precision": 1}
    if kind == "filter":
        precision = rng.choice([0, 1, 1])
        if rng.random() < 0.4:
            s = _log_int(rng, 9, 52 if precision else 20)
            nx, ny, nz = s, s + rng.randint(-2, 2), max(7, s // 2 + rng.randint(-1, 1))
            n = 3 * nx * ny * (nz - 1)
            k = min(n // 8, _log_int(rng, 9, 128 if precision else 40))
            precond = rng.choice([0, 1, 1])
            warm = rng.random() < 0.7
            return {"kind": kind, "grid": "elastic", "nx": nx, "ny": ny, "nz": nz, "k": k, "m": 8,
                    "it": rng.randint(8, 23 if precond and warm else 12), "precision": precision, "warm": warm,
                    "precond": precond}
        if rng.random() < 0.3:
            nx, ny, nz = _log_int(rng, 24, 200), _log_int(rng, 24, 200), 1
        else:
            s = _log_int(rng, 8, 44 if precision else 31)
            nx, ny, nz = s, s + rng.randint(-2, 2), s + rng.randint(-2, 2)
        k = min(nx * ny * nz // 8, _log_int(rng, 7, 170 if precision else 80))
        warm = rng.random() < 0.7
        return {"kind": kind, "grid": "scalar", "nx": nx, "ny": ny, "nz": nz, "k": k, "m": rng.choice([4, 8, 8, 16]),
                "it": rng.randint(5, 20 if warm else 12), "precision": precision, "warm": warm, "precond": 0}
    if kind == "apply":
        fp32 = rng.random() < 0.4
        if rng.random() < 0.5:
            s = _log_int(rng, 9, 40)
            return {"kind": kind, "grid": "elastic", "nx": s, "ny": s + rng.randint(-2, 2), "nz": max(3, s // 2),
                    "k": _log_int(rng, 8, 130), "fp32": fp32}
        s = _log_int(rng, 9, 44)
        return {"kind": kind, "grid": "scalar", "nx": s, "ny": s + rng.randint(-2, 2), "nz": s, "k": _log_int(rng, 8, 170),
                "fp32": fp32}
    if kind == "grad":
        if rng.random() < 0.35:
            s = rng.randint(8, 14)
            return {"kind": kind, "grid": "scalar", "nx": s, "ny": s - rng.randint(1, 2), "nz": s - rng.randint(2, 3),
                    "k": rng.randint(3, 16), "vectors": True}
        s = _log_int(rng, 9, 48)
        return {"kind": kind, "grid": rng.choice(["elastic", "scalar"]), "nx": s, "ny": s + rng.randint(-2, 2), "nz": s,
                "k": _log_int(rng, 3, 70), "vectors": False}
    precision = rng.choice([0, 1])
    s = _log_int(rng, 13, 41 if kind == "rr" else 21 if precision else 18)
    nx, ny, nz = s, s - rng.randint(0, 2), s - rng.randint(0, 2)
    if kind == "rr":
        return {"kind": kind, "grid": "scalar", "nx": nx, "ny": ny, "nz": nz, "k": _log_int(rng, 24, 170),
                "conv": rng.choice([0, 17, 40, 64])}
    want = rng.randint(20, 70 if precision else 40)
    return {"kind": kind, "grid": "scalar", "nx": nx, "ny": ny, "nz": nz, "k": -(-3 * want // 2), "want": want,
            "it": rng.randint(36, 48), "precision": precision}


# ------------------------------------------------------------------------------ pencils
def _axis(nodes, fixed, rng):
    """One axis: bands (n, 3) of the stiffness and mass matrices, and their eigenpairs."""
    if nodes == 1:
        return np.array([[0.0, 0.0, 0.0]]), np.array([[0.0, 1.0, 0.0]]), np.zeros(1), np.ones((1, 1))
    n = nodes + (1 if fixed else 0)  # nodes counts the free ones
    h = 1.0 / (n - 1)
    c = np.exp(rng.normal(0.0, 0.3, n - 1)) / h
    K, M = np.zeros((n, 3)), np.zeros((n, 3))
    K[:-1, 1] += c
    K[1:, 1] += c
    K[:-1, 2] -= c
    K[1:, 0] -= c
    M[:-1, 1] += h / 3
    M[1:, 1] += h / 3
    M[:-1, 2] += h / 6
    M[1:, 0] += h / 6
    if fixed:
        K, M = K[1:].copy(), M[1:].copy()
        K[0, 0] = M[0, 0] = 0.0

    def dense(b):
        return np.diag(b[:, 1]) + np.diag(b[:-1, 2], 1) + np.diag(b[1:, 0], -1)
    L = np.linalg.cholesky(dense(M))
    Li = np.linalg.inv(L)
    mu, Z = np.linalg.eigh(Li @ dense(K) @ Li.T)
    return K, M, mu, Li.T @ Z


class Pencil:
    """CSR pencil on the GPU; scalar boxes also know their one-dimensional eigenpairs."""

    def __init__(self, grid, nx, ny, nz, rng, want=None):
        self.grid, self.dims = grid, (nx, ny, nz)
        if grid == "elastic":
            self._elastic(nx, ny, nz, rng)
        else:
            self._scalar(nx, ny, nz, rng, want)
        self.n, self.nnz = self.rowptr.numel() - 1, self.col.numel()

    def _csr(self, cols, valid, a, b):
        """Rows of cols / valid / a / b, each (n, entries a row at most), to one CSR pattern."""
        cnt = valid.sum(1)
        self.rowptr = torch.zeros(cols.shape[0] + 1, dtype=torch.int64, device="cuda")
        torch.cumsum(cnt, 0, out=self.rowptr[1:])
        self.col = cols[valid].to(torch.int32)
        self.valA, self.valB = a[valid], b[valid]

    def _scalar(self, nx, ny, nz, rng, want):
        # with `want`, coefficients that leave a clear gap above that many eigenvalues
        for _ in range(40 if want else 1):
            self.axes = [_axis(s, d == 0, rng) for d, s in enumerate((nx, ny, nz))]
            if want and self.gap(want) >= 0.6 / want:
                break
        K = [torch.from_numpy(a[0]).cuda() for a in self.axes]
        M = [torch.from_numpy(a[1]).cuda() for a in self.axes]
        # axes of every array: z, y, x, then the offsets along z, y, x
        def spread(t, d):
            shape = [1] * 6
            shape[2 - d], shape[5 - d] = t.shape[0], 3
            return t.reshape(shape)
        Mx, My, Mz = (spread(M[d], d) for d in range(3))
        Kx, Ky, Kz = (spread(K[d], d) for d in range(3))
        b = Mz * My * Mx
        a = Mz * My * Kx + Mz * Ky * Mx + Kz * My * Mx + SHIFT * b
        valid, cols = self._neighbours(nx, ny, nz)
        n = nx * ny * nz
        self._csr(cols, valid, a.reshape(n, 27), b.reshape(n, 27))

    def _neighbours(self, nx, ny, nz):
        off = torch.arange(-1, 2, device="cuda")
        def ax(s, d):
            i = torch.arange(s, device="cuda")[:, None] + off[None, :]
            shape = [1] * 6
            shape[2 - d], shape[5 - d] = s, 3
            return i.reshape(shape)
        X, Y, Z = ax(nx, 0), ax(ny, 1), ax(nz, 2)
        valid = (X >= 0) & (X < nx) & (Y >= 0) & (Y < ny) & (Z >= 0) & (Z < nz)
        cols = X + nx * (Y + ny * Z)
        n = nx * ny * nz
        return valid.reshape(n, 27), cols.expand(valid.shape).reshape(n, 27)

    def _elastic(self, nx, ny, nz, rng):
        h = 1.0 / (max(nx, ny, nz) - 1)
        Ke, Me = (torch.from_numpy(t).cuda() for t in _brick(h, 0.3))
        gen = torch.Generator(device="cuda").manual_seed(int(rng.integers(1 << 31)))
        E = torch.exp(0.5 * torch.randn(nz - 1, ny - 1, nx - 1, 1, 1, generator=gen, dtype=torch.float64, device="cuda"))
        a = torch.zeros(nz, ny, nx, 27, 3, 3, dtype=torch.float64, device="cuda")
        b = torch.zeros_like(a)
        for l in range(8):
            lx, ly, lz = l & 1, (l >> 1) & 1, l >> 2
            at = (slice(lz, lz + nz - 1), slice(ly, ly + ny - 1), slice(lx, lx + nx - 1))
            for q in range(8):
                o = ((q & 1) - lx + 1) + 3 * (((q >> 1) & 1) - ly + 1) + 9 * ((q >> 2) - lz + 1)
                a[at][..., o, :, :] += E * Ke[3 * l:3 * l + 3, 3 * q:3 * q + 3]
                b[at][..., o, :, :] += Me[3 * l:3 * l + 3, 3 * q:3 * q + 3]
        valid, cols = self._neighbours(nx, ny, nz - 1)  # the free nodes: z >= 1
        nodes = nx * ny * (nz - 1)
        a, b = (t[1:].reshape(nodes, 27, 3, 3).permute(0, 2, 1, 3).reshape(3 * nodes, 81) for t in (a, b))
        valid = valid[:, None, :, None].expand(nodes, 3, 27, 3).reshape(3 * nodes, 81)
        cols = (3 * cols[:, None, :, None] + torch.arange(3, device="cuda")).expand(nodes, 3, 27, 3).reshape(3 * nodes, 81)
        self._csr(cols, valid, a, b)

    # scalar boxes: the lowest k eigenvalues and the axis indices of their eigenvectors
    def lowest(self, k):
        mx, my, mz = (a[2] for a in self.axes)
        lam = (mx[None, None, :] + my[None, :, None] + mz[:, None, None]).ravel() + SHIFT
        order = np.argsort(lam, kind="stable")[:k]
        nx, ny = len(mx), len(my)
        return lam[order], (order % nx, order // nx % ny, order // (nx * ny))

    def vectors(self, idx):
        """Eigenvectors (n, k), B-normalised, largest entry positive."""
        x, y, z = (torch.from_numpy(a[3][:, i].copy()).cuda() for a, i in zip(self.axes, idx))
        V = (z[:, None, None, :] * y[None, :, None, :] * x[None, None, :, :]).reshape(-1, x.shape[1])
        top = V.gather(0, V.abs().argmax(0, keepdim=True))
        return V * torch.sign(top)

    def gap(self, want):
        lam, _ = self.lowest(want + 1)
        return float(lam[want] / lam[want - 1] - 1)

    def interval(self, want):
        """gamma between the first `want` eigenvalues and the next one."""
        lam, _ = self.lowest(want + 1)
        return float(0.5 * (lam[want - 1] + lam[want]))

    def sparse(self, scale=None):
        A, B = self.valA, self.valB
        if scale is not None:
            s = scale.repeat_interleave(self.rowptr.diff()) * scale[self.col.long()]
            A, B = A * s, B * s
        ptr = self.rowptr.to(torch.int32)
        return tuple(torch.sparse_csr_tensor(ptr, self.col, v, size=(self.n, self.n)) for v in (A, B))

    def context(self, gamma, k, **opts):
        return slrf.Context(self.rowptr, self.col, self.valA, self.valB, gamma, k, slrf.slrf_opts_default(**opts))


def _brick(h, nu):
    """Stiffness (unit modulus) and mass (unit density) of a trilinear cube of side h, 24 x 24,
    dof 3 l + component, corner l = a + 2 b + 4 c; two Gauss points an axis."""
    lam, mu = nu / ((1 + nu) * (1 - 2 * nu)), 1.0 / (2 * (1 + nu))
    s = np.array([[2 * ((l >> d) & 1) - 1 for d in range(3)] for l in range(8)], dtype=float)
    K, M = np.zeros((8, 3, 8, 3)), np.zeros((8, 3, 8, 3))
    I, wt = np.eye(3), (h / 2) ** 3
    for p in np.ndindex(2, 2, 2):
        f = 1 + s * ((2 * np.array(p) - 1) / math.sqrt(3))
        N = f.prod(1) / 8
        dN = np.stack([s[:, d] * f[:, (d + 1) % 3] * f[:, (d + 2) % 3] for d in range(3)], 1) / (4 * h)
        M += wt * np.einsum("i,j,ab->iajb", N, N, I)
        K += wt * (lam * np.einsum("ia,jb->iajb", dN, dN) + mu * np.einsum("ib,ja->iajb", dN, dN)
                   + mu * np.einsum("ic,jc,ab->iajb", dN, dN, I))
    return K.reshape(24, 24), M.reshape(24, 24)


@functools.lru_cache(maxsize=None)
def _poles(m):
    """Shifted-Laplace poles and least-squares weights on the axis t / gamma."""
    x = (np.arange(m) + 0.5) / m
    s = x * (1 + 1j)
    t = np.concatenate([(np.arange(3000) + 0.5) / 3000, 1.3 * (51.0 / 1.3) ** (np.arange(3000) / 2999.0)])
    f = np.concatenate([np.ones(3000), np.zeros(3000)])
    c = 1.0 / (t[:, None] - s[None, :])
    G = np.concatenate([2 * c.real, -2 * c.imag], 1)
    G = np.concatenate([G, 0.1 * np.eye(2 * m)])
    y = np.linalg.lstsq(G, np.concatenate([f, np.zeros(2 * m)]), rcond=None)[0]
    return s, y[:m] + 1j * y[m:]


def _randn(seed, *shape):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(*shape, generator=g, dtype=torch.float64, device="cuda")


def _smooth(p, k):
    """The lowest Ritz pairs of an elasticity box in a space of low-frequency fields, zero on
    its clamped face: a block as the first outer steps leave it."""
    nx, ny, nz = p.dims
    def modes(s, cnt, clamp):
        t = torch.linspace(0, 1, s, dtype=torch.float64, device="cuda")[:, None]
        j = torch.arange(cnt, device="cuda")
        return torch.sin(math.pi * (j + 0.5) * t)[1:] if clamp else torch.cos(math.pi * j * t)
    Z, Y, X = modes(nz, 4, True), modes(ny, 4, False), modes(nx, 4, False)
    N = torch.einsum("za,yb,xc->zyxabc", Z, Y, X).reshape(-1, 64)
    V = torch.zeros(N.shape[0], 3, 3, 64, dtype=torch.float64, device="cuda")
    for a in range(3):
        V[:, a, a] = N
    V = V.reshape(p.n, 192)
    A, B = p.sparse()
    L = torch.linalg.cholesky(V.T @ (B @ V))
    H = torch.linalg.solve_triangular(L, V.T @ (A @ V), upper=False)
    H = torch.linalg.solve_triangular(L, H.T, upper=False)
    theta, S = torch.linalg.eigh(0.5 * (H + H.T))
    return (V @ torch.linalg.solve_triangular(L.T, S[:, :k], upper=True)).contiguous(), theta[:k].contiguous()


# ------------------------------------------------------------------------------ inputs
def _inputs(case, seed):
    """Pencil and blocks of a case (of each problem of a batch), from the seed alone."""
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    if kind == "batch":
        out = []
        for i in range(case["count"]):
            n = case["n_lo"] * (case["n_hi"] / case["n_lo"]) ** ((i + 0.5) / case["count"])
            s, want = round(n ** (0.5 if i % 2 else 1 / 3)), 10 + 3 * i
            p = Pencil("scalar", s, s - 1, 1 if i % 2 else s + 1, rng, want)
            L = -(-3 * want // 2)
            out.append((p, p.interval(want), want, L, _randn(seed + 1 + i, p.n, L)))
        return out
    p = Pencil(case["grid"], case["nx"], case["ny"], case["nz"], rng, case.get("want"))
    k = case["k"]
    d = {"pencil": p}
    if kind == "filter":
        s, w = _poles(case["m"])
        if case["grid"] == "elastic":
            d["X"], d["theta"] = _smooth(p, k)
            gamma = float(d["theta"][2 * k // 3])
        else:
            # Ritz block of an early outer step: eigenvectors with a hundredth of noise
            lam, idx = p.lowest(k)
            gamma = float(lam[max(0, 2 * k // 3 - 1)] * 1.001)
            V = p.vectors(idx)
            d["X"] = V + 0.01 * V.norm(dim=0) / math.sqrt(p.n) * _randn(seed, p.n, k)
            d["theta"] = torch.from_numpy(lam).cuda()
        if not case["warm"]:
            d["theta"] = None
        d["gamma"], d["sigma"], d["weights"] = gamma, s * gamma, w * gamma
    elif kind == "rr":
        lam, idx = p.lowest(case["conv"] + k)
        V = p.vectors(idx)
        d["gamma"] = float(lam[-1])
        d["locked"] = V[:, :case["conv"]].contiguous() if case["conv"] else None
        # a filtered block: damped eigenvectors, mixed, with a hundredth of noise
        W = V[:, case["conv"]:]
        mix = torch.eye(k, dtype=torch.float64, device="cuda") + 0.05 / math.sqrt(k) * _randn(seed + 1, k, k)
        damp = torch.linspace(1.0, 0.2, k, dtype=torch.float64, device="cuda")
        d["U"] = (W @ mix) * damp + 0.01 * V.norm() / math.sqrt(V.numel()) * _randn(seed, p.n, k)
    elif kind == "solve":
        d["gamma"] = p.interval(case["want"])
        d["X"] = _randn(seed, p.n, k)
    elif kind == "apply":
        d["X"] = _randn(seed, p.n, k)
    elif case["vectors"]:
        lam, idx = p.lowest(k)
        d["evals"], d["X"] = torch.from_numpy(lam).cuda(), p.vectors(idx)
        d["g"], d["gX"] = _randn(seed, k), _randn(seed + 1, p.n, k)
    else:
        d["X"] = _randn(seed, p.n, k) / math.sqrt(p.n)
        d["evals"] = _randn(seed + 1, k).abs().add(0.5).sort().values
        d["g"], d["gX"] = _randn(seed + 2, k), None
    return d


def prepare(case, seed):
    d = _inputs(case, seed)
    kind = case["kind"]
    if kind == "batch":
        opts = slrf.slrf_opts_default(precision=case["precision"], it_max=case["it"], it_adapt=1)
        b = slrf.Batch([(p.rowptr, p.col, p.valA, p.valB) for p, *_ in d], [g for _, g, *_ in d],
                       [L for *_, L, _ in d], opts)
        return {"kind": kind, "single": True, "batch": b, "V0": [v for *_, v in d]}
    p, k = d.pop("pencil"), case["k"]
    single = case.get("precision") == 1 or bool(case.get("fp32"))
    if kind == "filter":
        d["ctx"] = p.context(d["gamma"], k, m=case["m"], it_max=case["it"], precision=case["precision"],
                             precond=case["precond"], poles=d["sigma"], weights=d["weights"])
    elif kind == "rr":
        d["ctx"] = p.context(d["gamma"], max(k, case["conv"]))
        d["BX"] = None if d["locked"] is None else p.sparse()[1] @ d["locked"]
    elif kind == "solve":
        d["ctx"] = p.context(d["gamma"], k, it_max=case["it"], precision=case["precision"])
    elif kind == "apply":
        d["ctx"] = p.context(1.0, k, precision=int(case["fp32"]))
    else:
        d["ctx"] = p.context(1.0, k, tol_inner=1e-12)
    return {"kind": kind, "single": single, "fp32": case.get("fp32"), **d}


def run(s):
    kind = s["kind"]
    keep = (lambda t: t.float()) if s["single"] else (lambda t: t)
    if kind == "filter":
        return keep(s["ctx"].filter_apply(s["X"], s["theta"]))
    if kind == "rr":
        U, V, theta, res = s["ctx"].rayleigh_ritz(s["U"], s["locked"], s["BX"])
        return {"basis": U, "V": V, "theta": theta, "res": res}
    if kind == "solve":
        _, _, evals, X, _, _ = s["ctx"].solve(s["X"])
        return {"evals": evals, "X": X.float()}  # converged to 1e-8
    if kind == "batch":
        _, out, _ = s["batch"].solve(s["V0"])
        return [{"evals": evals, "X": X.float()} for _, _, evals, X, _ in out]
    if kind == "apply":
        AX, BX = s["ctx"].apply(s["X"], fp32=s["fp32"])
        return {"AX": keep(AX), "BX": keep(BX)}
    gA, gB = s["ctx"].eig_grad(s["evals"], s["X"], s["g"], s["gX"])
    return {"gA": gA, "gB": gB}


# ------------------------------------------------------------------------------ work
def _size(grid, nx, ny, nz):
    """Rows and stored entries of a box."""
    if grid == "elastic":
        return 3 * nx * ny * (nz - 1), 9 * math.prod(3 * s - 2 for s in (nx, ny, nz - 1))
    return nx * ny * nz, math.prod(3 * s - 2 if s > 1 else 1 for s in (nx, ny, nz))


def work(case):
    kind = case["kind"]
    if kind == "batch":
        # two outer steps at least, of It_max updates each, on blocks of 1.5 x 10 ... columns
        total = {"bytes": 0.0, "flops": 0.0}
        for i in range(case["count"]):
            n = case["n_lo"] * (case["n_hi"] / case["n_lo"]) ** ((i + 0.5) / case["count"])
            w = _filter_work(n, (9 if i % 2 else 27) * n, 15 + 3 * i, 8, case["it"], 8)
            total = {q: total[q] + 2 * w[q] for q in total}
        return total
    n, nnz = _size(case["grid"], case["nx"], case["ny"], case["nz"])
    k = case["k"]
    if kind == "filter":
        return _filter_work(n, nnz, k, case["m"], case["it"], 8 if case["precision"] else 16)
    if kind == "rr":
        c = case["conv"]
        # two passes against the locked block, two Gram matrices, the basis and the Ritz block
        flops = 2.0 * n * k * (4 * c + 2 * k + 3 * k) + 8.0 * nnz * k + 9.0 * k ** 3
        return {"bytes": 8.0 * n * (3 * k + 2 * c) + 20.0 * nnz, "flops": flops}
    if kind == "solve":
        w = _filter_work(n, nnz, k, 8, case["it"], 8 if case["precision"] else 16)
        return {q: 2 * v for q, v in w.items()}  # two outer steps at least
    if kind == "apply":
        return {"bytes": 24.0 * n * k + 20.0 * nnz, "flops": 4.0 * nnz * k}
    if case["vectors"]:
        # as many Lanczos steps as columns at least: one product and the vector recurrences
        return {"bytes": 8.0 * n * k * 2 + 36.0 * nnz, "flops": k * (4.0 * nnz * k + 20.0 * n * k)}
    return {"bytes": 8.0 * n * k + 20.0 * nnz, "flops": 4.0 * nnz * k}


def _filter_work(n, nnz, k, m, it, size):
    """The block in and out and the pencil once; every update reads and writes the residual,
    the direction and its image once.  8 operations per entry and complex column (A and B),
    about 40 per row and complex column for the recurrences and their sums."""
    state = n * k * m
    return {"bytes": 16.0 * n * k + (4 + size) * nnz + it * 6.0 * state * size,
            "flops": it * k * m * (8.0 * nnz + 40.0 * n)}


# ------------------------------------------------------------------------------ 64-bit results
def _exact_filter(p, X, theta, sigma, weights, it, tol, precond):
    """The COCG updates of every (pole, column) system in FP64."""
    dsc = None
    if precond:
        rows = torch.arange(p.n, device="cuda").repeat_interleave(p.rowptr.diff())
        diag = torch.zeros(p.n, dtype=torch.float64, device="cuda")
        on = rows == p.col
        diag[rows[on]] = p.valA[on]
        dsc = diag.rsqrt()
        del rows, on
    A0, B0 = p.sparse()
    A, B = p.sparse(dsc) if precond else (A0, B0)
    sig, wt = (torch.from_numpy(np.asarray(t)).cuda() for t in (sigma, weights))
    m, U = len(sigma), torch.empty_like(X)
    step = max(1, min(X.shape[1], int(1.5e9 // (16 * p.n * m))))
    for c0 in range(0, X.shape[1], step):
        V = X[:, c0:c0 + step]
        k = V.shape[1]
        if theta is None:
            g, c, U0 = B0 @ V, torch.ones(m, k, dtype=torch.complex128, device="cuda"), 0.0
        else:
            th = theta[c0:c0 + step]
            g = A0 @ V - th * (B0 @ V)
            c = 1.0 / (sig[:, None] - th[None, :])
            U0 = V * (2 * (wt[:, None] / (th[None, :] - sig[:, None])).real).sum(0)
        if dsc is not None:
            g = g * dsc[:, None]
        c, s = c.reshape(-1), sig.repeat_interleave(k)
        w = wt.repeat_interleave(k)

        def mul(r):
            flat = torch.view_as_real(r).reshape(p.n, -1)
            a, b = (torch.view_as_complex((M @ flat).reshape(p.n, -1, 2)) for M in (A, B))
            return a.sub_(b.mul_(s))

        def dot(a, b):  # unconjugated, in slices (no third block of this size)
            return sum((a[i:i + 65536] * b[i:i + 65536]).sum(0) for i in range(0, p.n, 65536))

        r = (g.repeat(1, m) * c).contiguous()
        pv, q = r.clone(), mul(r)
        acc = torch.zeros(p.n, k, dtype=torch.float64, device="cuda")
        rho, r0 = dot(r, r), dot(r.conj(), r).real
        live = r0 > 0
        mu = dot(pv, q)
        for i in range(it):
            al = torch.where(live, rho / mu, 0)
            acc += 2 * (pv * (w * al)).real.reshape(p.n, m, k).sum(1)
            r -= q * al
            new = dot(r, r)
            live = live & (dot(r.conj(), r).real > tol * tol * r0)
            if i + 1 == it or not bool(live.any()):
                break
            be = torch.where(live, new / rho, 0)
            rho = new
            pv = pv.mul_(be).add_(r)
            q = q.mul_(be).add_(mul(r))
            mu = dot(pv, q)
        U[:, c0:c0 + step] = U0 + (acc if dsc is None else acc * dsc[:, None])
    return U


def _exact_rr(p, U, locked):
    A, B = p.sparse()
    if locked is not None:
        BX = B @ locked
        for _ in range(2):
            U = U - locked @ (BX.T @ U)
    for _ in range(2):
        R = torch.linalg.cholesky(U.T @ (B @ U)).T
        U = torch.linalg.solve_triangular(R, U, upper=True, left=False)
    H = U.T @ (A @ U)
    theta, S = torch.linalg.eigh(0.5 * (H + H.T))
    V = U @ S
    V = V * torch.sign(V.gather(0, V.abs().argmax(0, keepdim=True)))
    AV = A @ V
    res = (AV - theta * (B @ V)).norm(dim=0) / AV.norm(dim=0)
    return {"basis": U, "V": V, "theta": theta, "res": res}


def _exact_pairs(p, count):
    lam, idx = p.lowest(count)
    return {"evals": torch.from_numpy(lam).cuda(), "X": p.vectors(idx)}


def _exact_grad(p, d):
    X, lam, g, gX = d["X"], d["evals"], d["g"], d["gX"]
    YA, YB = g * X, g * lam * X
    if gX is not None:
        _, B = p.sparse()
        rhs = -(gX - (B @ X) * (X * gX).sum(0))
        # solve in the eigenbasis of the box, one axis after the other
        Z = [torch.from_numpy(a[3].copy()).cuda() for a in p.axes]
        mx, my, mz = (torch.from_numpy(a[2].copy()).cuda() for a in p.axes)
        full = (mx[None, None, :] + my[None, :, None] + mz[:, None, None] + SHIFT)[..., None] - lam
        t = torch.einsum("zyxk,zc,yb,xa->cbak", rhs.reshape(*full.shape[:3], -1), Z[2], Z[1], Z[0])
        t = torch.where(full.abs() <= 1e-9 * lam, 0.0, t / full)
        xi = torch.einsum("cbak,zc,yb,xa->zyxk", t, Z[2], Z[1], Z[0]).reshape(p.n, -1)
        xi = xi - X * (X * (B @ xi)).sum(0)
        YA = YA + xi
        YB = YB + 0.5 * (gX * X).sum(0) * X + lam * xi
    rows = torch.arange(p.n, device="cuda").repeat_interleave(p.rowptr.diff())
    gA, gB = torch.empty_like(p.valA), torch.empty_like(p.valA)
    for i in range(0, p.nnz, 1 << 21):
        r, xc = rows[i:i + (1 << 21)], X[p.col[i:i + (1 << 21)].long()]
        gA[i:i + (1 << 21)] = (YA[r] * xc).sum(1)
        gB[i:i + (1 << 21)] = -(YB[r] * xc).sum(1)
    return {"gA": gA, "gB": gB}


def exact(case, seed):
    d = _inputs(case, seed)
    kind = case["kind"]
    if kind == "batch":
        return [_exact_pairs(p, count) for p, _, count, *_ in d]
    p = d["pencil"]
    if kind == "filter":
        return _exact_filter(p, d["X"], d["theta"], d["sigma"], d["weights"], case["it"], 1e-10, case["precond"])
    if kind == "rr":
        return _exact_rr(p, d["U"], d["locked"])
    if kind == "solve":
        return _exact_pairs(p, case["want"])
    if kind == "apply":
        A, B = p.sparse()
        return {"AX": A @ d["X"], "BX": B @ d["X"]}
    return _exact_grad(p, d)
