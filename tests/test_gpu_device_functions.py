"""Scalar device functions of csrc (common.cuh) against their definitions, element by element.

* norm_low, the norm of an FP32 panel column: the FP64 root rounded once to FP32, so it equals numpy's float32(sqrt(q))
  in every bit (IEEE 754 gives both operations one result).
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
