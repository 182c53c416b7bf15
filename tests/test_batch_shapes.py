"""The launch shapes a batch tries (CPU: the table alone): each once, within the kernels' most
threads per block, starting from the single-solve shape."""
import ctypes

import pytest


@pytest.fixture(scope="module")
def lib():
    from paper_2511_02700_gb300 import binding, build
    build.build()
    return binding.lib()


class FftShape(ctypes.Structure):
    _fields_ = [("units", ctypes.c_int), ("unit_threads", ctypes.c_int), ("max_threads", ctypes.c_int)]


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n", [8 << k for k in range(10)])
def test_trial_units(lib, n, prec):
    from paper_2511_02700_gb300 import binding as B
    shape = lib._ZN4pide9fft_shapeEii
    shape.restype = FftShape
    f = shape(2 * n, 8 if prec == B.PIDE2D_FP64 else 4)
    assert f.units >= 1 and f.unit_threads * f.units <= f.max_threads <= 1024
    assert 2 * n // f.unit_threads in (4, 8, 16) and 2 * n % f.unit_threads == 0
    out = (ctypes.c_int * 3)()
    k = lib._ZN4pide17batch_trial_unitsEiiPi(n, prec, out)
    got = list(out[:k])
    assert got == [u for u in (f.units, 2 * f.units, 4 * f.units) if u * f.unit_threads <= f.max_threads] and got
