"""Device bytes a handle asks for (gev_workspace_bytes, host arithmetic; no GPU).

A program may set ``workspace_limit`` to the bytes it has measured for its orders and options; a handle that fitted
such a limit has to fit it still, so the sizes may shrink but not grow."""
import ctypes
import glob
import os

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def L():
    if not glob.glob(os.path.join(ROOT, "paper_2502_02460_gb300", "_build", "libgev.so")):
        from paper_2502_02460_gb300 import build

        build.build()
    from paper_2502_02460_gb300 import gev

    return gev.lib()


def nbytes(L, n, dtype, prec, band_b):
    from paper_2502_02460_gb300 import gev

    o = gev.Opts()
    L.gev_default_opts(ctypes.byref(o))
    o.prec = prec
    o.band_b = band_b
    return L.gev_workspace_bytes(n, dtype, ctypes.byref(o))


@pytest.mark.parametrize("n,dtype,prec,band_b,most", [
    (300, 0, 0, 16, 29904896), (300, 0, 0, 64, 36113664), (300, 1, 1, 32, 55070208), (1000, 0, 0, 0, 137291776),
    (1000, 0, 1, 16, 151571968), (1000, 1, 0, 32, 250954240), (4096, 0, 0, 32, 1788654592), (4096, 0, 0, 0, 1804490752),
    (4096, 1, 1, 64, 5363512064)])
def test_workspace_does_not_grow(L, n, dtype, prec, band_b, most):
    assert nbytes(L, n, dtype, prec, band_b) <= most


@pytest.mark.parametrize("n,dtype,prec,default,widest", [(300, 0, 0, 16, 32), (1500, 0, 0, 32, 32), (2100, 0, 0, 32, 64),
                                                         (300, 1, 0, 16, 32), (2100, 1, 0, 32, 32), (2100, 0, 1, 32, 32)])
def test_room_for_wider_bands(L, n, dtype, prec, default, widest):
    """A width chosen by the table (negative band_b) leaves room for the bands that steps may ask for."""
    own, wide, auto = (nbytes(L, n, dtype, prec, b) for b in (default, widest, -default))
    assert auto >= wide >= own
    assert auto == own or widest > default
    assert nbytes(L, n, dtype, prec, -1) == nbytes(L, n, dtype, prec, 0)
