"""Paths chosen by size (short work, ragged edges, limits of a dispatch), at the sizes where they can go wrong.

* Divide and conquer: batched merge products (nodes up to 384 rows) and the parallel deflation scan with
  its rotation runs, on tridiagonals that deflate in every way (equal leaves, glued Wilkinson blocks, zero
  couplings).  Bound: the method is backward stable, 64 n eps ||T||_1 as for the other FP64 steps.
* Back-transform 2 reflector by reflector (16 columns per block, 8 lanes per column), at ragged windows and
  column counts, against the eigen-equation of the reduced matrix with the same bound.
* Its tensor-core form with prepared levels (orders with n k b >= 3e7), ragged levels and columns: same bound.
* Panels on both sides of the one-cluster limit: full -> band -> tridiagonal keeps trace and Frobenius norm to
  64 n eps of the latter.
* Emulated products whose K is shared by whole rounds of the SMs, and rows and columns whose exponents lie
  outside the middle of the range (the general output conversion): |err| <= K s_i t_j 2^-51 with the powers of two
  s_i, t_j above the largest entry of a row and a column (the scheme's normwise bound).
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


@pytest.mark.parametrize("n,k,b,cx", [(1037, 1000, 32, False), (901, 901, 64, False), (611, 600, 32, True), (703, 703, 16, True)])
def test_solve_with_prepared_levels(dev, n, k, b, cx):
    import torch

    from paper_2502_02460_gb300 import gev

    g = torch.Generator(device=dev)
    g.manual_seed(n)
    dt = torch.complex128 if cx else torch.float64
    H = torch.randn((n, n), generator=g, device=dev, dtype=dt)
    H = H + H.mH
    norm = float(H.abs().sum(dim=0).max())
    with gev.Solver(n, complex_=cx, device=dev, band_b=b) as s:
        w, C = s.solve(H, torch.eye(n, device=dev, dtype=dt), k)
    assert float((H @ C - C * w).abs().max()) <= 64 * n * EPS * norm
    assert float((C.mH @ C - torch.eye(k, device=dev, dtype=dt)).abs().max()) <= 64 * n * EPS


@pytest.mark.parametrize("n,b,cx", [(23, 16, False), (1440, 32, False), (2075, 64, False), (2430, 16, False), (505, 32, True),
                                    (830, 16, True), (740, 64, True)])
def test_to_tridiagonal_keeps_norms(dev, n, b, cx):
    import torch

    from paper_2502_02460_gb300 import gev

    g = torch.Generator(device=dev)
    g.manual_seed(n)
    A = torch.randn((n, n), generator=g, device=dev, dtype=torch.complex128 if cx else torch.float64)
    A = (A + A.mH).contiguous()
    trace, fro2 = float(A.diagonal().real.sum()), float((A.abs() ** 2).sum())
    with gev.Solver(n, complex_=cx, device=dev, band_b=b) as s:
        s.he2hb(gev.cm(A))
        d, e = s.hb2st()
    assert abs(float(d.sum()) - trace) <= 64 * n * EPS * fro2**0.5
    assert abs(float((d * d).sum() + 2 * (e * e).sum()) - fro2) <= 64 * n * EPS * fro2


@pytest.mark.parametrize("M,N,K,spread", [(9800, 64, 1000, 0), (130, 70, 5000, 0), (19500, 64, 300, 0), (300, 200, 77, 900),
                                          (260, 130, 700, 500)])
def test_emulated_product_shares_and_ranges(dev, M, N, K, spread):
    import ctypes

    import torch

    from paper_2502_02460_gb300 import gev

    L = gev.lib()
    L.gev_gemm_f64_scratch_bytes.restype = ctypes.c_size_t
    g = torch.Generator(device=dev)
    g.manual_seed(M + K)
    A = torch.randn((K, M), generator=g, device=dev, dtype=torch.float64)  # column-major M x K
    B = torch.randn((K, N), generator=g, device=dev, dtype=torch.float64)  # column-major N x K (op(B) = B^T)
    ea = torch.randint(-spread, spread + 1, (M,), generator=g, device=dev).to(torch.float64) // 2
    ref = A.T @ B
    A, B = A * torch.exp2(ea)[None, :], B * torch.exp2(-ea[:1]) if spread else B
    ref = (ref * torch.exp2(ea)[:, None] * torch.exp2(-ea[:1])) if spread else ref
    C = torch.empty((N, M), device=dev, dtype=torch.float64)
    nb = L.gev_gemm_f64_scratch_bytes(M, N, K)
    W = torch.empty(nb, dtype=torch.uint8, device=dev)
    st = torch.zeros(16, dtype=torch.int32, device=dev)
    p, d = (lambda t: ctypes.c_void_p(t.data_ptr())), ctypes.c_double
    stream = ctypes.c_void_p(torch.cuda.current_stream(dev).cuda_stream)
    rc = L.gev_gemm_f64(M, N, K, 0, 1, d(1.0), p(A), M, p(B), N, d(0.0), p(C), M, 1, stream, p(st), p(W), ctypes.c_size_t(nb))
    assert rc == 0
    s = torch.exp2(torch.floor(torch.log2(A.abs().amax(dim=0))) + 1)
    t = torch.exp2(torch.floor(torch.log2(B.abs().amax(dim=0))) + 1)
    assert bool(((C.T - ref).abs() <= K * s[:, None] * t[None, :] * 2.0**-51).all())


def test_mult_in_place(dev):
    """C = X^T Y into Y's own memory, at a size of the short products."""
    import torch

    from paper_2502_02460_gb300 import gev

    n, k = 100, 40
    g = torch.Generator(device=dev)
    g.manual_seed(1)
    X = torch.randn((n, n), generator=g, device=dev, dtype=torch.float64).tril()
    Y = torch.randn((n, k), generator=g, device=dev, dtype=torch.float64)
    Xb, Yb = gev.cm(X), gev.cm(Y)
    with gev.Solver(n, device=dev) as s:
        p = gev._ptr
        assert gev.lib().gev_step_mult(s.h, p(Xb), n, p(Yb), n, k, p(Yb), n) == 0
    assert float((Yb.T - X.T @ Y).abs().max()) <= 1e-13 * n * float((X.T @ Y).abs().max())


@pytest.mark.parametrize("emu", [0, 1])
@pytest.mark.parametrize("cx", [False, True])
@pytest.mark.parametrize("over", ["Y", "X", "Y shifted", "X shifted"])
@pytest.mark.parametrize("n,k", [(100, 40), (100, 100), (300, 200)])
def test_mult_over_an_operand(dev, n, k, over, cx, emu):
    """C = X^H Y into memory that holds Y or X (also from its middle on), with either engine, below and above the size of the
    short products (1.2e7 multiply-adds).  Bound: the emulated products' n s t (2^-52.6 + 2^-53 + n 2^-62.2) with
    s <= 2 max |X|, t <= 2 max |Y|, twice that for complex data's double inner dimension and sqrt(2) for its two parts."""
    import torch

    from paper_2502_02460_gb300 import gev

    g = torch.Generator(device=dev)
    g.manual_seed(n + k)
    dt = torch.complex128 if cx else torch.float64
    X = torch.randn((n, n), generator=g, device=dev, dtype=dt).tril()
    Y = torch.randn((n, k), generator=g, device=dev, dtype=dt)
    ref = X.mH @ Y
    mem = torch.zeros(2 * n * n + n * k + 7, dtype=dt, device=dev)  # X, then Y, then room behind it
    Xb, Yb = mem[: n * n].view(n, n), mem[n * n: n * n + n * k].view(k, n)
    Xb.copy_(X.T)
    Yb.copy_(Y.T)
    o = {"Y": n * n, "X": 0, "Y shifted": n * n + n + 7, "X shifted": n + 7}[over]
    Cb = mem[o: o + n * k].view(k, n)
    with gev.Solver(n, complex_=cx, device=dev, fp64_emulation=emu) as s:
        p = gev._ptr
        assert gev.lib().gev_step_mult(s.h, p(Xb), n, p(Yb), n, k, p(Cb), n) == 0
    bound = 16 * n * 2.0**-51 * float(X.abs().max()) * float(Y.abs().max())
    assert float((Cb.T - ref).abs().max()) <= bound


@pytest.mark.parametrize("cx", [False, True])
@pytest.mark.parametrize("n,k,width,b", [(300, 90, 64, 16), (300, 90, 64, 32), (37, 37, 32, 16), (1100, 700, 64, 16)])
def test_band_narrower_than_the_handles(dev, n, k, width, b, cx):
    """Reduction by steps with a narrower band than the handle's: its sweeps have more tasks.  Bound as above."""
    from paper_2502_02460_gb300 import gev

    rng = np.random.default_rng(n + b)
    A = rng.standard_normal((n, n)) + (1j * rng.standard_normal((n, n)) if cx else 0)
    A = A + A.conj().T
    norm = np.abs(A).sum(axis=0).max()
    with gev.Solver(n, complex_=cx, device=dev, band_b=width) as s:
        for bb in (b, width, b):  # the handle's own width in between
            assert s.he2hb(gev.cm_from_numpy(A, dev), bb) == bb
            d, e = s.hb2st()
            w, Z, _ = s.stedc(d, e, k)
            Y = gev.numpy_from_cm(s.back(Z, k))
            w = w.cpu().numpy()[:k]
            assert np.max(np.abs(A @ Y - Y * w)) <= 64 * n * EPS * norm
            assert np.max(np.abs(Y.conj().T @ Y - np.eye(k))) <= 64 * n * EPS


@pytest.mark.parametrize("n,b,cx", [(300, 32, False), (300, 32, True), (2100, 64, False), (2100, 16, False)])
def test_band_wider_than_the_tables_choice(dev, n, b, cx):
    """A handle whose width came from the table still reduces by steps to the bands that were its default.  Bound as above."""
    import torch

    from paper_2502_02460_gb300 import gev

    g = torch.Generator(device=dev)
    g.manual_seed(n + b)
    A = torch.randn((n, n), generator=g, device=dev, dtype=torch.complex128 if cx else torch.float64)
    A = A + A.mH
    norm, k = float(A.abs().sum(dim=0).max()), n // 7
    with gev.Solver(n, complex_=cx, device=dev) as s:
        own = s.band_b
        for bb in (b, own, b):
            assert s.he2hb(gev.cm(A), bb) == bb
            d, e = s.hb2st()
            w, Z, _ = s.stedc(d, e, k)
            Y = gev.logical(s.back(Z, k))
            assert float((A @ Y - Y * w[:k]).abs().max()) <= 64 * n * EPS * norm
            assert float((Y.mH @ Y - torch.eye(k, device=dev, dtype=A.dtype)).abs().max()) <= 64 * n * EPS


def test_band_limits_of_a_handle(dev):
    """An explicit width refuses wider bands; a limit at the explicit width's bytes still sets up a default handle."""
    import ctypes

    import torch

    from paper_2502_02460_gb300 import gev

    with gev.Solver(300, device=dev, band_b=16) as s:
        with pytest.raises(gev.GevError) as err:
            s.he2hb(torch.zeros((300, 300), dtype=torch.float64, device=dev), 32)
        assert err.value.code == 7
    for n, former in ((300, 32), (2100, 64)):
        o = gev.Opts()
        gev.lib().gev_default_opts(ctypes.byref(o))
        o.band_b = former
        limit = gev.lib().gev_workspace_bytes(n, gev.GEV_F64, ctypes.byref(o))
        with gev.Solver(n, device=dev, workspace_limit=limit) as s:
            A = torch.eye(n, dtype=torch.float64, device=dev)
            w, _ = s.solve_cm(2.0 * A, A, 3)
            assert float((w - 2.0).abs().max()) <= 64 * n * EPS


@pytest.mark.parametrize("M,N,K", [(130, 70, 40), (300, 65, 200)])
def test_emulated_product_at_the_ends_of_the_range(dev, M, N, K):
    """Rows scaled by powers of two so that outputs are subnormal, vanish or overflow.  The digits do not depend on the scale, so
    an output is that of the unscaled rows with another exponent, both rounded to nearest: within one unit in the last place
    (2^-1074 at least), infinite where that is.  General alpha and beta: the two further roundings, in every bit."""
    import ctypes

    import torch

    from paper_2502_02460_gb300 import gev

    L = gev.lib()
    L.gev_gemm_f64_scratch_bytes.restype = ctypes.c_size_t
    rng = np.random.default_rng(M)
    A0, B0 = rng.standard_normal((K, M)), rng.standard_normal((N, K))  # column-major op(A) = A0^T, op(B) = B0^T
    ea = rng.integers(-640, -560, M)                      # with 2^-440: subnormal and vanishing outputs
    up = np.arange(M) % 3 == 1
    ea[up] = rng.integers(715, 735, up.sum())             # with 2^300: finite and infinite outputs
    C0 = rng.standard_normal((N, M))
    nb = L.gev_gemm_f64_scratch_bytes(M, N, K)
    W = torch.empty(nb, dtype=torch.uint8, device=dev)
    st = torch.zeros(16, dtype=torch.int32, device=dev)
    p, d = (lambda t: ctypes.c_void_p(t.data_ptr())), ctypes.c_double
    stream = ctypes.c_void_p(torch.cuda.current_stream(dev).cuda_stream)

    def product(A, B, alpha, beta, C):
        A, B, C = (torch.from_numpy(np.ascontiguousarray(x)).to(dev) for x in (A, B, C))
        rc = L.gev_gemm_f64(M, N, K, 1, 0, d(alpha), p(A), K, p(B), K, d(beta), p(C), M, 1, stream, p(st), p(W),
                            ctypes.c_size_t(nb))
        assert rc == 0
        return C.cpu().numpy()

    A = np.ldexp(A0.T, ea[:, None])
    base = product(A0.T, B0, 1.0, 0.0, C0)
    low = product(A, np.ldexp(B0, -440), 1.0, 0.0, C0)
    high = product(A, np.ldexp(B0, 300), 1.0, 0.0, C0)
    with np.errstate(over="ignore", under="ignore"):
        want_low, want_high = np.ldexp(base, (ea - 440)[None, :]), np.ldexp(base, (ea + 300)[None, :])
    for got, want in ((low, want_low), (high, want_high)):
        fin = np.isfinite(want)
        assert np.array_equal(got[~fin], want[~fin]) and np.all(np.isfinite(got[fin]))
        assert np.all(np.abs(got[fin] - want[fin]) <= np.spacing(np.abs(want[fin])))
    assert np.any((low != 0) & (np.abs(low) < 2.0**-1022)) and np.any(low == 0)
    assert np.any(np.isinf(high)) and np.any(np.isfinite(high[:, up]))
    assert np.array_equal(product(A, np.ldexp(B0, -440), 1.5, 0.5, C0), 1.5 * low + 0.5 * C0)
