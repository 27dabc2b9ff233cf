"""The work that users of this library have it do, as timed cases.

Every case goes through the public calls of ``paper_2006_16117_gb300`` (the
Python binding of ``include/sim.h``) on finite-difference convection-diffusion
(-reaction) pencils, the operators of this repository's workloads and tests:

* ``apply``   y = (A - σB) x, the smallest call: residual checks of a user's own.
* ``solve``   x = (A - σB)^{-1} r for one shift: factorisation (or the
  separable preconditioner) and the refined inner solve.
* ``squares`` projected solves, residual and indicator of many squares against
  one given Krylov space.
* ``locate``  the whole method on one pencil: regions, levels, eigenvalues and,
  where asked for, multiplicities.
* ``batch``   the whole method on several pencils together.
* ``norm``    Φ = ||P f||² and its gradient on the stored entries (forward and
  adjoint solves at every node of a circle).
* ``eig``     a simple eigenvalue and its derivative on the stored entries.

``solver`` is ``band`` (a block factorisation per shift) or ``sep`` (the
fast-diagonalisation preconditioner); ``b`` is the kind of B: the identity, a
diagonal or a general matrix; ``precision`` is the handle's.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2006_16117_gb300 as S

BETA = (1.0, 0.5, 0.25)  # direction of the convection


# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the smallest call: one sparse apply on the 200×200 generalized pencil
        # (n = 40,000); latency and launches are all of it
        dict(name="apply_2d", kind="apply", ndim=2, grid=200, b="diag"),
        # one shifted solve on the small parity operator (n = 900), in FP64: a short
        # chain of small blocks, bound by launches and latencies
        dict(name="solve_small_fp64", kind="solve", ndim=2, grid=30, b="identity", solver="band", precision="fp64"),
        # one shifted solve on the benchmark's generalized pencil (n = 40,000) in
        # mixed precision: one long factorisation, then few refinement steps
        dict(name="solve_band_mixed", kind="solve", ndim=2, grid=200, b="diag", solver="band", precision="mixed"),
        # a general (tridiagonal) B and a grid that is no multiple of anything, FP64
        dict(name="solve_general_fp64", kind="solve", ndim=2, grid=97, b="general", solver="band", precision="fp64"),
        # one shifted solve of the 3-D reaction operator (n = 10^6) with the separable
        # preconditioner: the largest vectors, nothing factored
        dict(name="solve_sep_3d", kind="solve", ndim=3, grid=100, b="identity", solver="sep", precision="mixed"),
        # 4,096 squares against one Krylov space of dimension 50 (the evaluation of a level)
        dict(name="squares", kind="squares", m=50, count=4096),
        # the whole method with multiplicities on the small parity pencil, from a
        # fresh handle, as `run` does it: 50 closed-form eigenvalues
        dict(name="locate_small_fp64", kind="locate", ndim=2, grid=30, b="identity", solver="band", precision="fp64",
             count=50, multiplicity=True),
        # location on a slice of the benchmark pencil's region (n = 40,000, mixed)
        dict(name="locate_band_mixed", kind="locate", ndim=2, grid=200, b="diag", solver="band", precision="mixed",
             count=40, multiplicity=False),
        # location and multiplicities on a mid-size pencil (8 right-hand sides a shift)
        dict(name="locate_mult_mixed", kind="locate", ndim=2, grid=101, b="identity", solver="band",
             precision="mixed", count=60, multiplicity=True),
        # the 2-D reaction operator with the separable preconditioner: the low end of the spectrum
        dict(name="locate_sep_2d", kind="locate", ndim=2, grid=250, b="identity", solver="sep", precision="mixed",
             count=12, multiplicity=True),
        # six pencils of uneven size together, as parameter studies run them
        dict(name="batch", kind="batch", pencils=6, grid=60, precision="mixed", count=30),
        # differentiation through the projection on a band pencil: 16 nodes, forward and adjoint
        dict(name="norm_grad_band", kind="norm", ndim=2, grid=64, b="diag", solver="band", precision="fp64", nodes=16),
    ]


def draw(rng):
    log = lambda lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))  # noqa: E731
    kind = rng.choice(["apply", "solve", "solve", "solve", "squares", "locate", "locate", "batch", "norm", "eig"])
    prec = rng.choice(["fp64", "mixed"])
    if kind == "apply":
        nd = rng.choice([2, 3])
        return dict(kind=kind, ndim=nd, grid=log(30, 500) if nd == 2 else log(10, 100),
                    b=rng.choice(["identity", "diag", "general"]))
    if kind == "solve":
        solver = rng.choice(["band", "band", "sep"])
        if solver == "band":
            return dict(kind=kind, ndim=2, grid=log(20, 200 if prec == "mixed" else 140), solver=solver,
                        b=rng.choice(["identity", "diag", "general"]), precision=prec)
        nd = rng.choice([2, 3])
        return dict(kind=kind, ndim=nd, grid=log(30, 500) if nd == 2 else log(12, 100 if prec == "mixed" else 60),
                    solver=solver, b="identity", precision=prec)
    if kind == "squares":
        return dict(kind=kind, m=rng.randint(10, 52), count=log(64, 8192))
    if kind == "locate":
        if rng.random() < 0.7:
            return dict(kind=kind, ndim=2, grid=log(20, 110 if prec == "mixed" else 60), b=rng.choice(["identity", "diag"]),
                        solver="band", precision=prec, count=rng.randint(15, 40), multiplicity=rng.random() < 0.5)
        return dict(kind=kind, ndim=2, grid=log(40, 250 if prec == "mixed" else 100), b="identity", solver="sep",
                    precision=prec, count=rng.randint(6, 12), multiplicity=rng.random() < 0.5)
    if kind == "batch":
        return dict(kind=kind, pencils=rng.randint(2, 8), grid=log(16, 60), precision=prec, count=rng.randint(15, 30))
    if rng.random() < 0.5:
        return dict(kind=kind, ndim=2, grid=log(20, 64), b="identity" if kind == "eig" else rng.choice(["identity", "diag"]),
                    solver="band", precision=prec, nodes=rng.choice([8, 16]))
    return dict(kind=kind, ndim=2, grid=log(40, 300 if prec == "mixed" else 120), b="identity", solver="sep",
                precision=prec, nodes=rng.choice([8, 16]))


# ---------------------------------------------------------------------------
# operators
# ---------------------------------------------------------------------------
def _strength(seed, p=None):
    """The strength of the convection: the inputs' own, or pencil p's of a batch."""
    if p is None:
        return float(np.random.default_rng([seed, 11]).uniform(0.8, 1.6))
    return float(np.random.default_rng([seed, 13, p]).uniform(0.5, 5.0))


def _axes(N, ndim, pe):
    """(sub, diag, sup) of the central-difference operator along each axis."""
    h = 1.0 / (N + 1)
    return [(-1.0 / h**2 - pe * BETA[d] / (2 * h), 2.0 / h**2, -1.0 / h**2 + pe * BETA[d] / (2 * h))
            for d in range(ndim)]


def _axis_eigs(N, ax):
    k = np.arange(1, N + 1)
    return ax[1] + 2.0 * math.sqrt(ax[0] * ax[2]) * np.cos(k * math.pi / (N + 1))


def _spectrum(N, ndim, pe):
    """Sorted (real) eigenvalues of the separable part, B = I."""
    lam = np.zeros(1)
    for ax in _axes(N, ndim, pe):
        lam = (lam[:, None] + _axis_eigs(N, ax)[None, :]).reshape(-1)
    return np.sort(lam)


def _operator(N, ndim, pe, reaction):
    """-Δu + β·∇u + r u on an N^ndim grid, axis 0 fastest: CSR arrays."""
    n = N**ndim
    axes = _axes(N, ndim, pe)
    idx = np.arange(n, dtype=np.int64)
    diag = np.full(n, sum(a[1] for a in axes), dtype=np.complex128) + reaction
    cols, vals, keep = [], [], []
    for d in reversed(range(ndim)):
        i = (idx // N**d) % N
        cols.append(idx - N**d), vals.append(np.full(n, axes[d][0], dtype=np.complex128)), keep.append(i > 0)
    cols.append(idx), vals.append(diag), keep.append(np.ones(n, dtype=bool))
    for d in range(ndim):
        i = (idx // N**d) % N
        cols.append(idx + N**d), vals.append(np.full(n, axes[d][2], dtype=np.complex128)), keep.append(i < N - 1)
    keep = np.stack(keep, 1)
    indptr = np.concatenate([[0], np.cumsum(keep.sum(1))]).astype(np.int32)
    return indptr, np.stack(cols, 1)[keep].astype(np.int32), np.stack(vals, 1)[keep]


def _b_matrix(kind, n, rng):
    if kind == "identity":
        return None
    d = rng.uniform(1.0, 2.0, n).astype(np.complex128)
    if kind == "diag":
        return np.arange(n + 1, dtype=np.int32), np.arange(n, dtype=np.int32), d
    # a mass-matrix-like tridiagonal B
    idx = np.arange(n, dtype=np.int64)
    off = 0.2 * rng.uniform(0.5, 1.0, (n, 2))
    cols = np.stack([idx - 1, idx, idx + 1], 1)
    keep = np.stack([idx > 0, idx >= 0, idx < n - 1], 1)
    vals = np.stack([off[:, 0].astype(np.complex128), d, off[:, 1].astype(np.complex128)], 1)
    indptr = np.concatenate([[0], np.cumsum(keep.sum(1))]).astype(np.int32)
    return indptr, cols[keep].astype(np.int32), vals[keep]


def _gaussian(rng, n):
    return rng.standard_normal(n) + 1j * rng.standard_normal(n)


def _pencil(case, seed):
    """The case's pencil and its random generator (for what else it draws)."""
    rng = np.random.default_rng([seed, 17])
    N, ndim = case["grid"], case["ndim"]
    n = N**ndim
    reaction = np.zeros(n)
    if case.get("solver") == "sep":
        if ndim == 2:  # real reaction in [0, 1]
            reaction = rng.uniform(0.0, 1.0, n)
        else:          # complex reaction in the unit disk
            reaction = np.sqrt(rng.uniform(size=n)) * np.exp(2j * np.pi * rng.uniform(size=n))
    A = _operator(N, ndim, _strength(seed), reaction)
    B = _b_matrix(case.get("b", "identity"), n, rng)
    if case.get("b") == "diag":
        # A = B·(the operator), as a lumped mass matrix gives it: the operator's spectrum
        A = A[0], A[1], A[2] * np.repeat(B[2], np.diff(A[0]))
    return A, B, rng


def _window(lam, count, lo, hi):
    """The window of `count` neighbouring eigenvalues among lam[lo:hi] whose
    smallest gap (to the outer neighbours too) is largest: its real range."""
    best, at = -1.0, lo
    for s in range(max(lo, 1), max(max(lo, 1) + 1, min(hi, lam.size - count))):
        g = float(np.diff(lam[s - 1: s + count + 1]).min())
        if g > best:
            best, at = g, s
    return 0.5 * (lam[at - 1] + lam[at]), 0.5 * (lam[at + count - 1] + lam[at + count])


def _region(case, pe):
    N, ndim = case["grid"], case["ndim"]
    lam = _spectrum(N, ndim, pe)
    count = min(case["count"], lam.size // 3 - 2)
    if case.get("solver") == "sep":
        # the low end up to a gap that the reaction (in [0, 1]) cannot close
        c = count
        while lam[c] - lam[c - 1] <= 2.0:
            c += 1
        return float(lam[0] - 2.0), float(0.5 * (lam[c - 1] + 1.0 + lam[c])), -0.3, 0.7
    lo, hi = _window(lam, count, lam.size // 3, min(2 * lam.size // 3, lam.size // 3 + 400))
    return float(lo), float(hi), -0.3, 0.7


def _shift(case, seed):
    """A shift of the kind the method makes: inside the spectrum, at Im 0.2."""
    lam = _spectrum(case["grid"], case["ndim"], _strength(seed))
    at = lam[lam.size // 4]
    return complex(at / (1.44 if case["b"] == "general" else 1.0) + 0.5, 0.2)


def _options(case):
    # regions of dozens of eigenvalues need the shifts made inside the levels: without
    # them a square that no shift resolves can fill the last levels
    return S.sim_default_options(precision=case["precision"], new_shifts_in_levels=int(case["kind"] in ("locate", "batch")))


def _handle(case, seed, A, B):
    h = S.Sim(A, B, _options(case))
    if case["solver"] == "sep":
        h.set_separable((case["grid"],) * case["ndim"], _axes(case["grid"], case["ndim"], _strength(seed)))
    return h


def _batch_parts(case, seed):
    """Grid, strength of the convection and region of every pencil; the grids are the case's."""
    top, rng = case["grid"], np.random.default_rng(case["grid"] * 64 + case["pencils"])
    parts = []
    for p in range(case["pencils"]):
        N, pe = int(rng.integers(max(13, top // 2), top + 1)), _strength(seed, p)
        parts.append((N, pe, _region(dict(case, grid=N, ndim=2, b="identity"), pe)))
    return parts


def _circle(case, seed):
    """A circle around the smallest eigenvalue."""
    lam = _spectrum(case["grid"], case["ndim"], _strength(seed))
    return complex(lam[0] + 0.5, 0.0), 3.0


# ---------------------------------------------------------------------------
# what a user's program has in hand
# ---------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    if kind == "squares":
        H, centers, sides, sigma, beta = _square_inputs(case, seed)
        return dict(kind=kind, H=H, m=case["m"], centers=centers, sides=sides, sigma=sigma, beta=beta)
    if kind == "batch":
        rng = np.random.default_rng([seed, 23])
        parts = _batch_parts(case, seed)
        b = S.Batch([_operator(N, 2, pe, 0.0) for N, pe, _ in parts], None, _options(case))
        for p, (N, pe, _) in enumerate(parts):
            b.set_separable(p, (N, N), _axes(N, 2, pe))
        return dict(kind=kind, b=b, regions=[q[2] for q in parts], fs=[_gaussian(rng, q[0] * q[0]) for q in parts])
    A, B, rng = _pencil(case, seed)
    n = len(A[0]) - 1
    vec = _gaussian(rng, n)
    if kind == "apply":
        return dict(kind=kind, h=S.Sim(A, B), sigma=_shift(case, seed), x=torch.from_numpy(vec).cuda())
    if kind == "solve":
        return dict(kind=kind, h=_handle(case, seed, A, B), sigma=_shift(case, seed), r=torch.from_numpy(vec).cuda())
    if kind == "locate":
        st = dict(kind=kind, region=_region(case, _strength(seed)), f=vec, mult=case["multiplicity"], A=A, B=B, case=case)
        # small problems run from scratch in one call; larger ones keep their handle
        st["h"] = _handle(case, seed, A, B) if n > 5000 or case["solver"] == "sep" else None
        return st
    c, r = _circle(case, seed)
    return dict(kind=kind, h=_handle(case, seed, A, B), c=c, r=r, f=torch.from_numpy(vec).cuda(), nodes=case["nodes"],
                seed=seed, nnz=(len(A[1]), 0 if B is None else len(B[1])))


def run(st):
    kind = st["kind"]
    if kind == "apply":
        return st["h"].apply_shifted(st["sigma"], st["x"])
    if kind == "solve":
        return st["h"].shifted_solve(st["sigma"], st["r"])[0]
    if kind == "squares":
        return S.eval_squares(st["H"], st["m"], st["beta"], st["sigma"], st["centers"], st["sides"])
    if kind == "locate":
        if st["h"] is None:
            eig, mult, _ = S.run(st["A"], st["B"], st["region"], st["f"], _options(st["case"]), st["mult"])
            return (eig, mult) if st["mult"] else (eig,)
        h = st["h"]
        h.set_region(st["region"], st["f"])
        h.solve_all_levels()
        eig = h.eigenvalues()
        return (eig, h.multiplicity()) if st["mult"] else (eig,)
    if kind == "batch":
        b = st["b"]
        b.set_regions(st["regions"], st["fs"])
        b.solve_all_levels()
        return [b.eigenvalues(p) for p in range(b.count)]
    if kind == "norm":
        phi = st["h"].projection_norm(st["c"], st["r"], st["f"], st["nodes"])
        gA, gB = st["h"].projection_norm_grad(*st["nnz"], device=True)
        return (phi, gA) if gB is None else (phi, gA, gB)
    lam, dA, _ = st["h"].eigenvalue_grad(st["c"], st["r"], st["nnz"][0], nodes=st["nodes"], seed=st["seed"], device=True)
    return np.array([lam]), dA


def _square_inputs(case, seed):
    """A Krylov space's Hessenberg matrix as the method meets it: m Ritz values
    of M = (A - σB)^{-1}B spread around σ, and squares of side 1/4 and smaller
    around the eigenvalues σ + 1/d near it."""
    rng = np.random.default_rng([seed, 29])
    m, count = case["m"], case["count"]
    # d_k = 1 / (λ_k - σ) with λ_k - σ between 0.5 and a few hundred either side
    gap = np.cumsum(rng.uniform(0.5, 6.0, m)) * np.where(np.arange(m) % 2 == 0, 1.0, -1.0)
    d = 1.0 / (gap - 0.2j)
    M = np.diag(d) + np.triu(0.02 * _gaussian(rng, m * m).reshape(m, m), 1) * np.abs(d)[None, :]
    # Arnoldi on a unitarily mixed copy gives an unreduced Hessenberg matrix
    Q0, _ = np.linalg.qr(_gaussian(rng, m * m).reshape(m, m))
    M = Q0 @ M @ Q0.conj().T
    V = np.zeros((m, m), dtype=np.complex128)
    H = np.zeros((m + 1, m), dtype=np.complex128)
    v = _gaussian(rng, m)
    V[:, 0] = v / np.linalg.norm(v)
    for j in range(m):
        w = M @ V[:, j]
        for _ in range(2):
            c = V[:, : j + 1].conj().T @ w
            H[: j + 1, j] += c
            w = w - V[:, : j + 1] @ c
        H[j + 1, j] = np.linalg.norm(w) if j + 1 < m else 1e-4
        if j + 1 < m:
            V[:, j + 1] = w / H[j + 1, j]
    sigma = complex(1000.0, 0.2)
    lam = sigma + gap - 0.2j
    sides = 0.25 * 2.0 ** -rng.integers(0, 10, count).astype(np.float64)
    centers = lam[rng.integers(0, m, count)] + 2.0 * sides * (rng.uniform(-1, 1, count) + 1j * rng.uniform(-1, 1, count))
    return H, centers, sides, sigma, float(rng.uniform(0.5, 2.0))


# ---------------------------------------------------------------------------
# what one pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    kind = case["kind"]
    if kind == "squares":
        m, c = case["m"], case["count"]
        # eight triangular solves a square (m²/2 complex multiply-adds each)
        return {"bytes": 16.0 * m * (m + 1) + 40.0 * c, "flops": 32.0 * m * m * c}
    if kind == "batch":
        shifts = 1 + case["count"] // 12
        parts = [_work_locate(q[0] * q[0], q[0], 5, shifts, False, "sep", 2, 8) for q in _batch_parts(case, 0)]
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    N, nd = case["grid"], case["ndim"]
    n = N**nd
    nnz = (2 * nd + 1) * n
    if kind == "apply":
        nb = {"identity": 0, "diag": 16 * n, "general": 60 * n}[case["b"]]
        return {"bytes": 20.0 * nnz + nb + 32.0 * n, "flops": 8.0 * nnz}
    cs = 8 if case["precision"] == "mixed" else 16
    if kind == "solve":
        by, fl = _work_solve(n, N, nnz, case["solver"], nd, cs, 1)
        return {"bytes": by, "flops": fl}
    if kind == "locate":
        shifts = 1 + case["count"] // 12
        by, fl = _work_locate(n, N, 2 * nd + 1, shifts, case["multiplicity"], case["solver"], nd, cs)
        return {"bytes": by, "flops": fl}
    by, fl = _work_solve(n, N, nnz, case["solver"], nd, cs, 1)
    k = 2 * case["nodes"]
    return {"bytes": k * by + 16.0 * nnz, "flops": k * (fl + 8.0 * nnz)}


def _work_solve(n, N, nnz, solver, nd, cs, solves):
    """One factorisation (written once) and `solves` solves through it."""
    if solver == "sep":
        return 20.0 * nnz + 32.0 * n * solves, solves * (16.0 * n * N * nd + 8.0 * nnz)
    T, nb = N, N
    fac = 2.0 * nb * T * T
    return fac * cs + 20.0 * nnz + solves * (fac * cs + 32.0 * n), 8.0 * nb * T**3 + solves * (8.0 * fac + 8.0 * nnz)


def _work_locate(n, N, per_row, shifts, mult, solver, nd, cs):
    m = 50
    by = fl = 0.0
    for jobs in (1, 8) if mult else (1,):
        b, f = _work_solve(n, N, per_row * n, solver, nd, cs, m + 1)
        by += shifts * (b + jobs * (m + 1) * 16.0 * n)
        fl += shifts * (f + (m + 1) * (jobs - 1) * 16.0 * N * n + jobs * 16.0 * (m * m / 2) * n)
    return by, fl


# ---------------------------------------------------------------------------
# the same in 64 bits, without the library
# ---------------------------------------------------------------------------
def _sparse(M, n):
    if M is None:
        i = torch.arange(n)
        return torch.sparse_coo_tensor(torch.stack([i, i]), torch.ones(n, dtype=torch.complex128), (n, n))
    indptr, indices, data = M
    rows = np.repeat(np.arange(n), np.diff(indptr))
    return torch.sparse_coo_tensor(torch.from_numpy(np.stack([rows, indices]).astype(np.int64)),
                                   torch.from_numpy(np.ascontiguousarray(data)), (n, n))


def _entries(M, n):
    """Rows, columns and values of the stored entries."""
    if M is None:
        return np.arange(n), np.arange(n), np.ones(n, dtype=np.complex128)
    return np.repeat(np.arange(n), np.diff(M[0])), M[1].astype(np.int64), M[2]


def _times(rows, cols, vals, x):
    out = np.zeros(x.size, dtype=np.complex128)
    p = vals * x[cols]
    out.real = np.bincount(rows, p.real, x.size)
    out.imag = np.bincount(rows, p.imag, x.size)
    return out


class _BlockSolver:
    """LU of a matrix whose entries couple neighbouring blocks of T rows only
    (block elimination with dense pivoted LUs), with iterative refinement."""

    def __init__(self, rows, cols, vals, n, T):
        self.e = (rows, cols, vals)
        self.n, self.T, self.nb = n, T, -(-n // T)
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        order = np.argsort(rows, kind="stable")
        r, c, v = rows[order], cols[order], vals[order]
        at = np.searchsorted(r, np.arange(self.nb + 1) * T)
        self.lu, self.up, self.low = [], [], []
        prev = None
        for k in range(self.nb):
            rk, ck, vk = r[at[k]: at[k + 1]] - k * T, c[at[k]: at[k + 1]] - (k - 1) * T, v[at[k]: at[k + 1]]
            W = np.zeros((T, 3 * T), dtype=np.complex128)
            np.add.at(W, (rk, ck), vk)
            for i in range(max(0, n - k * T), T):
                W[i, T + i] = 1.0
            W = torch.from_numpy(W).to(dev)
            L, D, U = W[:, :T].contiguous(), W[:, T: 2 * T].contiguous(), W[:, 2 * T:].contiguous()
            if prev is not None:
                D = D - L @ torch.linalg.lu_solve(*prev, self.up[-1])
            prev = torch.linalg.lu_factor(D)
            self.lu.append(prev), self.up.append(U), self.low.append(L)
        self.dev = dev

    def _once(self, b):
        T = self.T
        x = torch.zeros(self.nb * T, 1, dtype=torch.complex128, device=self.dev)
        x[: self.n, 0] = torch.from_numpy(b).to(self.dev)
        t = []
        for k in range(self.nb):
            rhs = x[k * T: (k + 1) * T]
            if k:
                rhs = rhs - self.low[k] @ t[-1]
            t.append(torch.linalg.lu_solve(*self.lu[k], rhs))
        for k in range(self.nb - 2, -1, -1):
            t[k] = t[k] - torch.linalg.lu_solve(*self.lu[k], self.up[k] @ t[k + 1])
        return torch.cat(t)[: self.n, 0].cpu().numpy()

    def solve(self, b):
        x = self._once(b)
        for _ in range(2):
            x = x + self._once(b - _times(*self.e, x))
        return x


def _shifted_entries(A, B, n, z):
    ra, ca, va = _entries(A, n)
    rb, cb, vb = _entries(B, n)
    return np.concatenate([ra, rb]), np.concatenate([ca, cb]), np.concatenate([va, -z * vb])


def exact(case, seed):
    kind = case["kind"]
    if kind == "squares":
        return _exact_squares(case, seed)
    if kind == "batch":
        return [_closed_form(N, 2, pe, region) for N, pe, region in _batch_parts(case, seed)]
    if kind == "locate":
        if case["solver"] == "sep":
            return None
        pe = _strength(seed)
        eig = _closed_form(case["grid"], case["ndim"], pe, _region(case, pe))
        return (eig, None) if case["multiplicity"] else (eig,)
    N, nd = case["grid"], case["ndim"]
    A, B, rng = _pencil(case, seed)
    n = N**nd
    vec = _gaussian(rng, n)
    if kind == "apply":
        return _times(*_shifted_entries(A, B, n, _shift(case, seed)), vec)
    T = N ** (nd - 1)
    if T > 200:
        return None
    if kind == "solve":
        return _BlockSolver(*_shifted_entries(A, B, n, _shift(case, seed)), n, T).solve(vec)
    if kind == "eig" or N > 128:
        return None
    c, r = _circle(case, seed)
    K = case["nodes"]
    w = r * np.exp(2j * np.pi * np.arange(K) / K) / K
    xs = [_BlockSolver(*_shifted_entries(A, B, n, c + K * w[j]), n, T).solve(vec) for j in range(K)]
    p = sum(w[j] * xs[j] for j in range(K))
    ra, ca, va = _entries(A, n)
    rb, cb, vb = _entries(B, n)
    gA, gB = np.zeros(ra.size, dtype=np.complex128), np.zeros(rb.size, dtype=np.complex128)
    for j in range(K):
        rows, cols, vals = _shifted_entries(A, B, n, c + K * w[j])
        mu = _BlockSolver(cols, rows, vals.conj(), n, T).solve(np.conj(w[j]) * p)
        gA -= 2.0 * mu[ra] * xs[j][ca].conj()
        gB += 2.0 * np.conj(c + K * w[j]) * mu[rb] * xs[j][cb].conj()
    phi = float(np.vdot(p, p).real)
    return (phi, gA) if B is None else (phi, gA, gB)


def _closed_form(N, ndim, pe, region):
    lam = _spectrum(N, ndim, pe)
    return lam[(lam >= region[0]) & (lam <= region[1])].astype(np.complex128)


def _exact_squares(case, seed):
    """Indicator and largest residual of every square by dense solves."""
    H, centers, sides, sigma, beta = _square_inputs(case, seed)
    m = case["m"]
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    Hm = torch.from_numpy(H[:m]).to(dev)
    eye = torch.eye(m, dtype=torch.complex128, device=dev)
    rhs = torch.zeros(m, 1, dtype=torch.complex128, device=dev)
    rhs[0, 0] = beta
    u = torch.from_numpy(np.exp(2j * np.pi * np.arange(8) / 8)).to(dev)
    ind, rho = [], []
    for a in range(0, case["count"], 1024):
        c = torch.from_numpy(centers[a: a + 1024]).to(dev)
        rad = torch.from_numpy(sides[a: a + 1024]).to(dev) / math.sqrt(2.0)
        off = rad[:, None] * u[None, :]
        alpha = sigma - (c[:, None] + off)
        y = torch.linalg.solve(eye + alpha[:, :, None, None] * Hm, rhs.expand(c.numel(), 8, m, 1))[..., 0]
        fine = (off[:, :, None] * y).sum(1) / 8
        coarse = (off[:, ::2, None] * y[:, ::2]).sum(1) / 4
        ind.append(fine.norm(dim=1) / coarse.norm(dim=1))
        rho.append((alpha.abs() * abs(H[m, m - 1]) * y[..., -1].abs() / y.norm(dim=2)).max(1).values)
    return torch.cat(ind), torch.cat(rho)
