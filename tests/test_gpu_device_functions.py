"""Scalar device functions of csrc (common.cuh, int_sums.cuh) against their definitions, element by element.

* norm_low, the norm of an FP32 panel column: the FP64 root rounded once to FP32, so it equals numpy's float32(sqrt(q))
  in every bit (IEEE 754 gives both operations one result).
* recip and recip_sqrt, against CUDA's division and rsqrt and against extended precision.  In units of u = 2^-53 relative:
  the hardware's start takes 20 bits of the mantissa and returns 20, 2^-18.4 at most, so the series' cut is below
  2^-55.2 = 0.22 u and recip errs by its last rounding and the cut, 1.25 u; recip_sqrt by the rounding of q y, which enters by
  half, the last one and the cut (5/16 e^3): 1.75 u.  Outside the exponents of the steps, zero, subnormals, infinities and
  NaN included, they are CUDA's own results in every bit.
* house (reflector scalars) against their definitions in extended precision, with q's roundings 1 u (complex 3 u) entering
  r = 1 / sqrt(q) by half.  Real: beta = q r 3.25 u; tau = 1 + |alpha| r, at most 2, 4.25 u absolute; scale = s r / tau 6.7 u.
  Complex: beta 4.25 u; tau 8.2 u absolute; scale = conj(d) / |d|^2 with d = alpha - beta to 5.25 u, |d|^2 to 12.5 u:
  scale (alpha - beta) within 26.5 u of 1.
* sum_block against exact sums: each of the N values is cut to 57 bits below the largest exponent, less than 2^-56 of the
  largest value, and the total is rounded once; where the largest exponent is near either end it is the plain sum, in every bit.
* to_fp64, (acc 2^-49 + sh) 2^e with sh cut to units of 2^-81, against the exact value rounded once to nearest even, in every
  bit, from subnormal results to overflow; to_fp64_fast, for the middle of the range, to half an ulp and the rounding of
  sh's fraction, in units of 2^-49: 2^-25 in FP32 and 2^-32 of its integer form.
"""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def fns(tmp_path_factory):
    import torch

    from paper_2502_02460_gb300 import build

    assert torch.cuda.is_available()
    so = str(tmp_path_factory.mktemp("fns") / "device_functions.so")
    cmd = [build.nvcc(), *build.ARCH, *build.NVFLAGS, "--extended-lambda", "-shared", "-cudart", "shared",
           os.path.join(HERE, "device_functions.cu"), "-o", so]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(so)


def call(f, ins, out_dtype, out_shape=None):
    """out = f(inputs), numpy arrays through device memory."""
    import torch

    dev = torch.device("cuda:0")
    ins = [torch.from_numpy(np.ascontiguousarray(a)).to(dev) for a in ins]
    out = torch.from_numpy(np.empty(out_shape or ins[0].shape, dtype=out_dtype)).to(dev)
    torch.cuda.synchronize()
    n = out.shape[0]
    assert f(ctypes.c_int(n), *[ctypes.c_void_p(a.data_ptr()) for a in ins], ctypes.c_void_p(out.data_ptr())) == 0
    return out.cpu().numpy()


def test_norm_of_an_fp32_column(fns):
    rng = np.random.default_rng(0)
    q = rng.uniform(1.0, 4.0, 100000) * 2.0 ** rng.integers(-240, 240, 100000)
    q = np.concatenate([q, (1.0 + 2.0**-24) ** 2 * 4.0 ** np.arange(-60.0, 60.0), [2.0**-298, 1e76, 0.0]])
    assert np.array_equal(call(fns.t_norm_low, [q], np.float32), np.sqrt(q).astype(np.float32))


def _sweep(lo, hi, per, seed, negative):
    """Finite doubles with biased exponents lo .. hi, per each: random mantissas, mantissas at both ends, signs."""
    rng = np.random.default_rng(seed)
    e = np.repeat(np.arange(lo, hi + 1, dtype=np.uint64), per)
    m = rng.integers(0, 1 << 52, e.size, dtype=np.uint64)
    k = np.arange(e.size) % per
    m[k == 0], m[k == 1], m[k == 2], m[k == 3] = 0, 1, (1 << 52) - 1, 1 << 51
    x = ((e << np.uint64(52)) | m).view(np.float64)
    return np.where(rng.random(e.size) < 0.5, -x, x) if negative else x


SPECIAL = np.array([0.0, -0.0, 5e-324, -5e-324, 2.0**-1022, 1.7976931348623157e308, np.inf, -np.inf, np.nan])


def _exact(x):
    """x in extended precision: longdouble has 64 bits here or 113 on Arm."""
    return x.astype(np.longdouble)


def test_recip(fns):
    x = np.concatenate([_sweep(24, 2020, 64, 1, True), _sweep(1021, 1026, 20000, 2, True)])
    y = call(fns.t_recip, [x], np.float64)
    assert np.max(np.abs(_exact(x) * _exact(y) - 1)) <= 1.25 * 2.0**-53
    div = call(fns.t_divide, [x], np.float64)
    assert np.max(np.abs(y - div) / np.spacing(np.abs(div))) <= 1
    out = np.concatenate([_sweep(0, 23, 64, 3, True), _sweep(2021, 2046, 64, 4, True), SPECIAL])
    assert np.array_equal(call(fns.t_recip, [out], np.float64), call(fns.t_divide, [out], np.float64), equal_nan=True)


def test_recip_sqrt(fns):
    x = np.concatenate([_sweep(24, 2020, 64, 5, False), _sweep(1021, 1026, 20000, 6, False)])
    y = call(fns.t_recip_sqrt, [x], np.float64)
    assert np.max(np.abs(_exact(y) * np.sqrt(_exact(x)) - 1)) <= 1.75 * 2.0**-53
    cuda = call(fns.t_rsqrt, [x], np.float64)
    assert np.max(np.abs(y - cuda) / np.spacing(cuda)) <= 3  # 1.75 ulp here, CUDA's documented 1 ulp there
    out = np.concatenate([_sweep(0, 23, 64, 7, False), _sweep(2021, 2046, 64, 8, False), SPECIAL[SPECIAL >= 0], [np.nan]])
    assert np.array_equal(call(fns.t_recip_sqrt, [out], np.float64), call(fns.t_rsqrt, [out], np.float64), equal_nan=True)


def _columns(n, seed):
    rng = np.random.default_rng(seed)
    xn = rng.random(n) * 2.0 ** rng.integers(-60, 60, n)
    xn[: n // 8] = 0.0  # (complex data: a rotation of alpha only)
    return rng, xn


def test_house_real(fns):
    n = 50000
    rng, xn = _columns(n, 9)
    al = rng.standard_normal(n) * 2.0 ** rng.integers(-40, 40, n)
    al[-100:] = 0.0
    tau, beta, scale = call(fns.t_house, [al, xn], np.float64, (n, 3)).T
    a = _exact(al)
    s = np.where(np.signbit(al), -1, 1)
    nrm = np.sqrt(a * a + _exact(xn))
    b = -s * nrm
    u = 2.0**-53
    assert np.max(np.abs(beta - b) / nrm) <= 4 * u
    assert np.max(np.abs(tau - (b - a) / b)) <= 5 * u
    assert np.max(np.abs(_exact(scale) * (a - b) - 1)) <= 7 * u


def test_house_complex(fns):
    n = 50000
    rng, xn = _columns(n, 10)
    al = (rng.standard_normal(n) + 1j * rng.standard_normal(n)) * 2.0 ** rng.integers(-40, 40, n)
    al[-100:] = 0.0
    o = call(fns.t_house_cx, [al, xn], np.float64, (n, 6))
    o = _exact(o)
    x, y = _exact(al.real), _exact(al.imag)
    s = np.where(al.real >= 0, 1, -1)
    nrm = np.sqrt(x * x + y * y + _exact(xn))
    u = 2.0**-53
    assert np.max(np.abs(o[:, 2] + s * nrm) / nrm) <= 5 * u and not np.any(o[:, 3])
    # tau = (beta - alpha) / beta = 1 + s alpha / nrm, |tau| <= 2
    assert np.max(np.hypot(o[:, 0] - (1 + s * x / nrm), o[:, 1] - s * y / nrm)) <= 9 * u
    # scale (alpha - beta) = 1
    dx, dy = x + s * nrm, y
    assert np.max(np.hypot(o[:, 4] * dx - o[:, 5] * dy - 1, o[:, 4] * dy + o[:, 5] * dx)) <= 27 * u


@pytest.mark.parametrize("N", [20, 40])
def test_sum_block(fns, N):
    rng = np.random.default_rng(N)
    n = 4000
    v = rng.standard_normal((n, N)) * 2.0 ** rng.integers(-30, 30, (n, N)) * 2.0 ** rng.integers(-900, 900, (n, 1))
    v[:500] *= 2.0 ** rng.integers(-60, 1, (500, N))   # far apart
    v[500:1000, 1:N:2] = -v[500:1000, 0:N:2]           # cancels exactly
    v[1000:1200, :] = 0.0
    v[1200:1400, 3:] = 0.0
    v[1400:1800] = np.sign(v[1400:1800]) * np.repeat(rng.uniform(1.0, 2.0, (400, 1)), N, 1)  # equal magnitudes
    v[1800:1900] = 1.9999999999999998                  # the largest carry
    base = np.ldexp(rng.uniform(1.0, 2.0, (800, N)), rng.integers(-20, 0, (800, N)))
    base[:, 0] = 1.5
    for q, biased in enumerate([0, 1, 99, 100, 101, 2000, 2001, 2040]):  # exponents at the limits
        v[2000 + 100 * q:2100 + 100 * q] = np.ldexp(base[100 * q:100 * q + 100], biased - 1023)
    v[2900, 0], v[2901, 1], v[2902, 2] = np.inf, np.nan, -np.inf
    f = getattr(fns, f"t_sum_block_{N}")
    out = call(f, [v], np.float64, (n,))
    top = ((v.view(np.int64) >> 52) & 0x7FF).max(axis=1)
    mid = (top >= 100) & (top <= 2000)
    with np.errstate(all="ignore"):
        plain = np.zeros(n)
        for u in range(N):
            plain = plain + v[:, u]
    assert np.array_equal(out[~mid], plain[~mid], equal_nan=True) and mid.sum() > 3000 and (~mid).sum() > 500
    for i in np.flatnonzero(mid):
        exact = sum(map(Fraction, v[i]))
        bound = N * Fraction(2) ** -56 * Fraction(np.abs(v[i]).max()) + Fraction(np.spacing(abs(out[i]))) / 2
        assert abs(Fraction(out[i]) - exact) <= bound
    assert np.array_equal(call(f, [v[mid][:, ::-1]], np.float64, (int(mid.sum()),)), out[mid])  # any order


def _accumulators(n, seed):
    """(acc, sh) as the product kernel forms them: |acc| < 2^62, |sh| < 2^-18; ties and carries of every width among them."""
    rng = np.random.default_rng(seed)
    acc = rng.integers(-(1 << 62), 1 << 62, n) >> rng.integers(0, 62, n)
    sh = (rng.uniform(-1.0, 1.0, n) * 2.0 ** -rng.integers(18, 90, n)).astype(np.float32)
    sh[::5] = 0.0
    k = rng.integers(1, 10, n)
    tie = np.arange(n) % 5 == 0  # acc = odd or even mantissa and exactly half a unit, or all ones
    acc[tie] = (((rng.integers(1 << 52, 1 << 53, n) << 1) + 1) << (k - 1) >> rng.integers(0, 2, n))[tie]
    acc[7::50] = (1 << 62) - 1
    acc[8::50] = -(1 << 53) + 1
    acc[9::50] = 0
    acc[10::50], sh[10::50] = 0, 0.0
    return rng, acc, sh


def _shifted(total, k):
    """total 2^k rounded once to FP64 (CPython's integer division and conversion round to nearest even)."""
    try:
        return float(total << k) if k >= 0 else total / (1 << -k)
    except OverflowError:
        return np.inf if total > 0 else -np.inf


def test_to_fp64_rounds_once(fns):
    n = 60000
    rng, acc, sh = _accumulators(n, 11)
    e = np.concatenate([rng.integers(-1140, 1140, n // 3), rng.integers(-1090, -1010, n // 3), rng.integers(-20, 20, n // 3)])
    e = e.astype(np.int32)
    out = call(fns.t_to_fp64, [acc, sh, e], np.float64, (n,))
    want = np.empty(n)
    for i in range(n):
        low = Fraction(float(sh[i])) * 2**81
        si = abs(low).__floor__() * (1 if low >= 0 else -1)
        want[i] = _shifted((int(acc[i]) << 32) + si, int(e[i]) - 81)
    assert np.array_equal(out, want)
    sub = (np.abs(want) < 2.0**-1022) & (want != 0)
    assert sub.sum() > 3000 and np.isinf(want).sum() > 300


def test_to_fp64_fast(fns):
    n = 40000
    rng, acc, sh = _accumulators(n, 12)
    e = rng.integers(-800, 801, n).astype(np.int32)
    out = call(fns.t_to_fp64_fast, [acc, sh, e], np.float64, (n,))
    for i in range(n):
        scale = Fraction(2) ** int(e[i])
        exact = (Fraction(int(acc[i]), 1 << 49) + Fraction(float(sh[i]))) * scale * (-1 if i & 1 else 1)
        assert abs(Fraction(out[i]) - exact) <= Fraction(np.spacing(abs(out[i]))) / 2 + scale * (Fraction(2) ** -74 + Fraction(2) ** -81)
