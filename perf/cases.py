"""Work that users of this solver have it do, as cases that can be timed and compared.

A case is a dict of plain values.  ``prepare`` builds what a program holds before the call (the pencil on
the GPU in the library's column-major layout, a handle), ``run`` is one pass through the public entry
points of ``paper_2502_02460_gb300.gev``, ``work`` counts what the path cannot do without and ``exact``
gives the results in 64 bits without this repository's code.

Pencils.  S = L L^H with L a lower-triangular band of decaying entries (localised basis functions whose
overlaps vanish beyond a cutoff radius), H = L (Q diag(lambda) Q^H) L^H with Q orthogonal / unitary and a
DFT-like spectrum: 10 % core levels in [-100, -10], 40 % valence in [-1, 0], 50 % conduction in [0.5, 5],
each evenly spread with a random jitter (a gapped system; no two levels coincide, so the single vectors
are determined).  The exact eigenvectors are C = L^-H Q.  Q is a product of random signs and fast Hartley
(complex: Fourier) transforms, dense and cheap to build on the GPU at any order.
"""
from __future__ import annotations

import math

import torch

from paper_2502_02460_gb300 import gev

CUTOFF = 24  # sub-diagonals of L


def listed():
    return [
        # smallest serving request: one small molecule, all pairs; latency and launches count
        {"name": "solve_real_256_all", "kind": "solve", "n": 256, "k": 256, "complex": False, "mixed": False,
         "reuse": False},
        # one SCF iteration of a small k-point (odd basis size): the factor of S is resident
        {"name": "solve_complex_509_scf", "kind": "solve", "n": 509, "k": 128, "complex": True, "mixed": False,
         "reuse": True},
        # a full SCF step of a mid-size system: the eigenpairs, then both density matrices
        {"name": "solve_density_real_1500", "kind": "scf", "n": 1500, "k": 375, "complex": False},
        # a k-point of a periodic system, k = N/4 as in the serving stream
        {"name": "solve_complex_2048", "kind": "solve", "n": 2048, "k": 512, "complex": True, "mixed": False,
         "reuse": False},
        # the N = 4096 configuration with 30 % of the pairs
        {"name": "solve_real_4096", "kind": "solve", "n": 4096, "k": 1229, "complex": False, "mixed": False,
         "reuse": False},
        # the largest plain solve: above the one-stage range, k = N/4
        {"name": "solve_real_10240", "kind": "solve", "n": 10240, "k": 2560, "complex": False, "mixed": False,
         "reuse": False},
        # mixed precision, the occupied half of the spectrum, small
        {"name": "mixed_real_1000", "kind": "solve", "n": 1000, "k": 500, "complex": False, "mixed": True,
         "reuse": False},
        # mixed precision, large
        {"name": "mixed_real_6144", "kind": "solve", "n": 6144, "k": 3072, "complex": False, "mixed": True,
         "reuse": False},
        # mixed precision, complex k-point
        {"name": "mixed_complex_1536", "kind": "solve", "n": 1536, "k": 768, "complex": True, "mixed": True,
         "reuse": False},
        # the reduction to the standard problem through the step entry points: factor, inverse, A = X H X^H
        {"name": "standard_form_real_5000", "kind": "standard", "n": 5000, "complex": False},
        # density and energy-weighted density matrix of given orbitals
        {"name": "density_complex_3000", "kind": "density", "n": 3000, "k": 750, "complex": True},
        # ill-conditioned overlap: the pencil in the eigenbasis of S, 100 directions omitted
        {"name": "reduced_real_1200", "kind": "reduced", "n": 1200, "m": 1100, "k": 300},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "mixed", "mixed", "scf", "standard", "density", "reduced"])
    cx = rng.random() < 0.4
    if kind == "solve":
        n = _log_int(rng, 200, 3000 if cx else 9000)
        k = max(1, int(n * rng.choice([0.25, 0.25, 0.3, 0.5, 1.0] if n < 5000 else [0.25, 0.3])))
        return {"kind": "solve", "n": n, "k": k, "complex": cx, "mixed": False, "reuse": rng.random() < 0.5}
    if kind == "mixed":
        n = _log_int(rng, 500, 1800 if cx else 6000)
        return {"kind": "solve", "n": n, "k": _occupied(n), "complex": cx, "mixed": True, "reuse": rng.random() < 0.3}
    if kind == "scf":
        n = _log_int(rng, 300, 3000)
        return {"kind": "scf", "n": n, "k": max(1, n // 4), "complex": cx}
    if kind == "standard":
        return {"kind": "standard", "n": _log_int(rng, 300, 3000 if cx else 7000), "complex": cx}
    if kind == "density":
        n = _log_int(rng, 400, 4000 if cx else 9000)
        return {"kind": "density", "n": n, "k": max(1, n // 4), "complex": cx}
    n = _log_int(rng, 300, 1600)
    m = n - max(1, n // rng.randint(8, 16))
    return {"kind": "reduced", "n": n, "m": m, "k": max(1, m // 4)}


# ------------------------------------------------------------------------------------- pencils --
def _gen(seed, dev):
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    return g


def _occupied(n):
    return int(round(0.1 * n)) + int(round(0.4 * n))


def _spread(lo, hi, m, g, dev):
    u = torch.rand(m, generator=g, device=dev, dtype=torch.float64)
    i = torch.arange(m, device=dev, dtype=torch.float64)
    return lo + (i + 0.2 + 0.6 * u) / max(m, 1) * (hi - lo)


def _spectrum(n, g, dev):
    n_core, n_val = int(round(0.1 * n)), int(round(0.4 * n))
    return torch.cat([_spread(-100.0, -10.0, n_core, g, dev), _spread(-1.0, 0.0, n_val, g, dev),
                      _spread(0.5, 5.0, n - n_core - n_val, g, dev)])


class _Q:
    """A dense random orthogonal (unitary) operator: signs (phases), transform, signs, transform, signs."""

    def __init__(self, n, cx, g, dev):
        self.n, self.cx = n, cx
        if cx:
            u = torch.rand((3, n), generator=g, device=dev, dtype=torch.float64) * (2.0 * math.pi)
            self.d = torch.polar(torch.ones_like(u), u)
        else:
            self.d = torch.randint(0, 2, (3, n), generator=g, device=dev).to(torch.float64) * 2.0 - 1.0

    def _transform(self, X):
        F = torch.fft.fft(X, dim=0)
        if not self.cx:
            F = F.real - F.imag
        return F.mul_(1.0 / math.sqrt(self.n))

    def apply(self, X):
        X = self._transform(self.d[2][:, None] * X)
        X = self._transform(self.d[1][:, None] * X)
        return self.d[0][:, None] * X

    def dense(self, dev):
        return self.apply(torch.eye(self.n, device=dev, dtype=self.d.dtype))


def _coeffs(cx):
    if cx:
        return [1.0] + [0.5 * math.exp(-0.4 * j) * complex(math.cos(0.2 * j), math.sin(0.2 * j))
                        for j in range(1, CUTOFF + 1)]
    return [1.0] + [0.5 * math.exp(-0.5 * j) * math.cos(0.3 * j) for j in range(1, CUTOFF + 1)]


def _apply_l(X, cx):
    """L X for the banded lower-triangular L."""
    a = _coeffs(cx)
    Y = X.clone()
    for j in range(1, min(CUTOFF, X.shape[0] - 1) + 1):
        Y[j:] += a[j] * X[:-j]
    return Y


def _dense_l(n, cx, dev):
    return _apply_l(torch.eye(n, device=dev, dtype=torch.complex128 if cx else torch.float64), cx)


def _herm(X):
    return (X + X.mH).mul_(0.5)


def _congruence(apply_left, X):
    """F X F^H for the operator F and a Hermitian X."""
    return _herm(apply_left(apply_left(X).mH))


def _pencil(n, cx, seed, dev):
    """(H, S) as logical matrices, and the levels and the operator Q."""
    g = _gen(seed, dev)
    lam = _spectrum(n, g, dev)
    q = _Q(n, cx, g, dev)
    M = _congruence(q.apply, torch.diag(lam.to(q.d.dtype)))
    H = _congruence(lambda X: _apply_l(X, cx), M)
    L = _dense_l(n, cx, dev)
    S = _congruence(lambda X: _apply_l(X, cx), torch.eye(n, device=dev, dtype=L.dtype))
    return H, S, lam, q


def _levels(n, cx, seed, dev):
    g = _gen(seed, dev)
    lam = _spectrum(n, g, dev)
    return lam, _Q(n, cx, g, dev)


def _orbitals(n, cx, q, k, dev):
    """C = L^-H Q, the first k columns."""
    return torch.linalg.solve_triangular(_dense_l(n, cx, dev).mH, q.dense(dev)[:, :k], upper=True)


def _phase(C):
    """The library's convention: the entry of largest modulus of each column is real and positive."""
    i = C.abs().argmax(dim=0)
    p = C.gather(0, i[None, :])
    return C * (p.conj() / p.abs())


def _occupations(k, seed, dev):
    """Fractional occupations of a finite-temperature SCF step."""
    u = torch.rand(k, generator=_gen(seed + 7, dev), device=dev, dtype=torch.float64)
    return 2.0 - 0.5 * u * u


def _reduced_parts(n, m, k, seed, dev):
    """Overlap with n - m negligible eigenvalues: its eigenbasis U, the kept sigma, levels and Q."""
    g = _gen(seed, dev)
    U = _Q(n, False, g, dev)
    sigma = _spread(0.1, 3.0, m, g, dev)
    lam = _spread(-10.0, 5.0, m, g, dev)
    q = _Q(m, False, g, dev)
    return U, sigma, lam, q


# --------------------------------------------------------------------------------- the protocol --
def prepare(case, seed):
    dev = torch.device("cuda")
    kind, n, cx = case["kind"], case["n"], case.get("complex", False)
    st = {"kind": kind, "k": case.get("k", n)}
    st["solver"] = gev.Solver(n, complex_=cx, mixed=case.get("mixed", False))
    if kind == "density":
        lam, q = _levels(n, cx, seed, dev)
        st["C"] = gev.cm(_orbitals(n, cx, q, case["k"], dev))
        st["w"] = lam[: case["k"]].contiguous()
        st["occ"] = _occupations(case["k"], seed, dev)
        return st
    if kind == "reduced":
        m = case["m"]
        U, sigma, lam, q = _reduced_parts(n, m, case["k"], seed, dev)
        M = _congruence(q.apply, torch.diag(lam))
        sh = sigma.sqrt()
        core = torch.zeros((n, n), device=dev, dtype=torch.float64)
        core[:m, :m] = sh[:, None] * M * sh[None, :]
        core[m:, m:] = torch.eye(n - m, device=dev, dtype=torch.float64)
        st["H"] = gev.cm(_congruence(U.apply, core))
        tail = torch.tensor([1e-9, 1e-12, 0.0], device=dev, dtype=torch.float64).repeat((n - m) // 3 + 1)[: n - m]
        st["S"] = gev.cm(_congruence(U.apply, torch.diag(torch.cat([sigma, tail]))))
        return st
    H, S, _, _ = _pencil(n, cx, seed, dev)
    st["H"], st["S"] = gev.cm(H), gev.cm(S)
    if kind == "scf":
        st["occ"] = _occupations(case["k"], seed, dev)
    if case.get("reuse"):  # an SCF cycle under way: the first iteration left the factor of S in the handle
        st["solver"].reuse_factor(True)
        st["solver"].solve_cm(st["H"], st["S"], case["k"])
        st["S"] = None
    return st


def run(st):
    s, k, kind = st["solver"], st["k"], st["kind"]
    if kind == "solve":
        w, C = s.solve_cm(st["H"], st["S"], k)
        return {"w": w, "C": C}
    if kind == "scf":
        w, C = s.solve_cm(st["H"], st["S"], k)
        P, PE = s.density(C, st["occ"], w)
        return {"w": w, "C": C, "P": P, "PE": PE}
    if kind == "density":
        P, PE = s.density(st["C"], st["occ"], st["w"])
        return {"P": P, "PE": PE}
    if kind == "reduced":
        w, C, m = s.solve_reduced_cm(st["H"], st["S"], 1e-5, k)
        return {"w": w, "C": C, "m": m}
    L = st["S"].clone()
    s.potrf(L)
    X = L.clone()
    s.trtri(X)
    A = s.hegst(st["H"], X)
    return {"L": L, "X": X, "A": A}


def work(case):
    """Inputs read once and outputs written once; floating-point operations of the reduction (Cholesky and
    inverse 2/3 n^3, A = X H X^H n^3, tridiagonalisation 4/3 n^3, back-transform 2 n^2 k, C = X^H Y n^2 k),
    of the orbital products n^2 k per density matrix; complex operations count four times."""
    n, kind = case["n"], case["kind"]
    cx = case.get("complex", False)
    es, f = (16, 4.0) if cx else (8, 1.0)
    k = case.get("k", n)
    if kind == "solve":
        flops = (2.0 / 3.0 if not case["reuse"] else 0.0) * n**3 + 7.0 / 3.0 * n**3 + 3.0 * n * n * k
        return {"bytes": es * ((1 if case["reuse"] else 2) * n * n / 2 + n * k) + 8 * k, "flops": f * flops}
    if kind == "scf":
        return {"bytes": es * (n * n + n * k + 2 * n * n) + 16 * k, "flops": f * (3.0 * n**3 + 5.0 * n * n * k)}
    if kind == "density":
        return {"bytes": es * (n * k + 2 * n * n) + 16 * k, "flops": f * 2.0 * n * n * k}
    if kind == "standard":
        return {"bytes": es * (n * n + 2.5 * n * n), "flops": f * 5.0 / 3.0 * n**3}
    m = case["m"]
    flops = 4.0 / 3.0 * n**3 + 2.0 * n * n * m + 2.0 * n * n * m + n * m * m + 4.0 / 3.0 * m**3 + 2.0 * m * m * k + 2.0 * n * m * k
    return {"bytes": 8 * (n * n + n * k) + 8 * k, "flops": flops}


def exact(case, seed):
    dev = torch.device("cuda")
    kind, n, cx = case["kind"], case["n"], case.get("complex", False)
    if kind == "reduced":
        m, k = case["m"], case["k"]
        U, sigma, lam, q = _reduced_parts(n, m, k, seed, dev)
        Y = torch.zeros((n, k), device=dev, dtype=torch.float64)
        Y[:m] = q.dense(dev)[:, :k] / sigma.sqrt()[:, None]
        return {"w": lam[:k], "C": _phase(U.apply(Y)).T.contiguous(), "m": m}
    lam, q = _levels(n, cx, seed, dev)
    if kind == "standard":
        L = _dense_l(n, cx, dev)
        X = torch.linalg.solve_triangular(L, torch.eye(n, device=dev, dtype=L.dtype), upper=False)
        M = _congruence(q.apply, torch.diag(lam.to(q.d.dtype)))
        return {"L": L.T.contiguous(), "X": X.T.contiguous(), "A": M.T.contiguous()}
    k = case["k"]
    C = _orbitals(n, cx, q, k, dev)
    w = lam[:k]
    if kind == "solve":
        return {"w": w, "C": _phase(C).T.contiguous()}
    out = {"w": w, "C": _phase(C).T.contiguous()} if kind == "scf" else {}
    occ = _occupations(k, seed, dev)
    # P_ij = sum_l f_l conj(C_il) C_jl: its column-major buffer holds P_ij at [j, i]
    out["P"] = (C * occ) @ C.mH
    out["PE"] = (C * (occ * w)) @ C.mH
    return out
