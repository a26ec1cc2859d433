"""The paths taken by short work, at the sizes where they can go wrong.

* Divide and conquer: batched merge products (nodes up to 384 rows) and the parallel deflation scan with
  its rotation runs, on tridiagonals that deflate in every way (equal leaves, glued Wilkinson blocks, zero
  couplings).  Bound: the method is backward stable, 64 n eps ||T||_1 as for the other FP64 steps.
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
