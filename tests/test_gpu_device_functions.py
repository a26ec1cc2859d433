"""Scalar device functions of csrc (common.cuh) against their definitions, element by element.

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
"""
import ctypes
import os
import subprocess

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
