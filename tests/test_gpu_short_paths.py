"""The paths taken by short work, at the sizes where they can go wrong.

* Divide and conquer: batched merge products (nodes up to 384 rows) and the parallel deflation scan with
  its rotation runs, on tridiagonals that deflate in every way (equal leaves, glued Wilkinson blocks, zero
  couplings).  Bound: the method is backward stable, 64 n eps ||T||_1 as for the other FP64 steps.
* Back-transform 2 reflector by reflector (16 columns per block, 8 lanes per column), at ragged windows and
  column counts, against the eigen-equation of the reduced matrix with the same bound.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
EPS = np.finfo(float).eps


@pytest.fixture(scope="module")
def dev():
    import torch

    from paper_2502_02460_gb300 import build

    build.build()
    return torch.device("cuda:0")


def _tridiag(kind, n):
    rng = np.random.default_rng(n)
    if kind == "equal":  # equal leaves, weak couplings: runs of rotations at every merge
        d = np.tile(rng.standard_normal(8), n // 8 + 1)[:n]
        e = np.tile(rng.standard_normal(8), n // 8 + 1)[: n - 1]
        e[::8] = 1e-14
    elif kind == "wilkinson":
        d = np.abs(np.arange(n) % 21 - 10.0)
        e = np.ones(n - 1)
        e[20::21] = 1e-9
    elif kind == "zeros":
        d = rng.standard_normal(n)
        e = rng.standard_normal(n - 1)
        e[::5] = 0.0
    else:
        d = rng.standard_normal(n)
        e = rng.standard_normal(n - 1)
    return d, e


@pytest.mark.parametrize("kind", ["random", "equal", "wilkinson", "zeros"])
@pytest.mark.parametrize("n", [2, 32, 33, 100, 384, 385, 770])
def test_stedc_deflation(dev, n, kind):
    import torch

    from paper_2502_02460_gb300 import gev

    d, e = _tridiag(kind, n)
    T = np.diag(d) + np.diag(e, 1) + np.diag(e, -1)
    norm = np.abs(T).sum(axis=0).max()
    for k in (n, max(1, n // 3)):
        with gev.Solver(n, device=dev) as s:
            w, Z, _ = s.stedc(torch.from_numpy(d).to(dev), torch.from_numpy(e).to(dev), k)
            w, Z = w.cpu().numpy(), gev.numpy_from_cm(Z)
        assert np.all(np.diff(w) >= 0)
        assert np.max(np.abs(w - np.linalg.eigvalsh(T))) <= 64 * n * EPS * norm
        assert np.max(np.abs(T @ Z - Z * w[:k])) <= 64 * n * EPS * norm
        assert np.max(np.abs(Z.T @ Z - np.eye(k))) <= 64 * n * EPS


@pytest.mark.parametrize("emu", [0, 1])
@pytest.mark.parametrize("cx", [False, True])
@pytest.mark.parametrize("n,k,b", [(3, 3, 16), (18, 1, 16), (65, 17, 32), (97, 16, 64), (130, 129, 64), (259, 33, 32)])
def test_two_stage_back(dev, n, k, b, cx, emu):
    from paper_2502_02460_gb300 import gev

    rng = np.random.default_rng(n + b)
    A = rng.standard_normal((n, n)) + (1j * rng.standard_normal((n, n)) if cx else 0)
    A = A + A.conj().T
    norm = np.abs(A).sum(axis=0).max()
    with gev.Solver(n, complex_=cx, device=dev, band_b=b, fp64_emulation=emu) as s:
        s.he2hb(gev.cm_from_numpy(A, dev))
        d, e = s.hb2st()
        w, Z, _ = s.stedc(d, e, k)
        Y = gev.numpy_from_cm(s.back(Z, k))
        w = w.cpu().numpy()[:k]
    assert np.max(np.abs(A @ Y - Y * w)) <= 64 * n * EPS * norm
    assert np.max(np.abs(Y.conj().T @ Y - np.eye(k))) <= 64 * n * EPS
