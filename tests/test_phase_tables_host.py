"""The host's phase tables for the FP32 and double-float kernels (every eighth entry
evaluated, the others products) against 80-bit arithmetic.

Bound, in units of u = 2^-53 of the scale: cosine and sine 0.6 each and one rounding
of their correction, for both factors; one rounding of the scaling; three of the
product's component: below 10 u.  The rounding of gamma c alone would be up to
|gamma c| u, 800 u at the largest entries here."""
import ctypes

import numpy as np
import pytest

from paper_2401_02852_gb300 import _lib

L = np.longdouble
if np.finfo(L).nmant < 63:
    pytest.skip("needs an extended-precision long double", allow_module_level=True)


def _table(gamma, scale, m, arith):
    f = _lib.load()["_ZN4qaoa11phase_tableEddiiPdS0_"]
    f.restype = None
    f.argtypes = [ctypes.c_double, ctypes.c_double, ctypes.c_int, ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p]
    re, im = np.zeros(m + 1), np.zeros(m + 1)
    f(gamma, scale, m, arith, re.ctypes.data, im.ctypes.data)
    return re, im


@pytest.mark.parametrize("arith", [0, 2])  # FP32, double-float
@pytest.mark.parametrize("m", [0, 1, 7, 8, 9, 128, 255])
@pytest.mark.parametrize("gamma", [0.0, 0.04, -0.31, 0.8, 1.57, -3.2, 3.14159])
def test_entries(arith, m, gamma):
    scale = 2.0 ** -7.5
    re, im = _table(gamma, scale, m, arith)
    x = L(gamma) * np.arange(m + 1).astype(L)
    err = np.maximum(np.abs(re - L(scale) * np.cos(x)), np.abs(im + L(scale) * np.sin(x)))
    assert float(err.max()) <= 10 * 2.0 ** -53 * scale


@pytest.mark.parametrize("arith", [0, 2])
@pytest.mark.parametrize("gamma", [1e5, 2.5e5, 2.7e5, 1e9, 1e17, 1e300])
def test_huge_angles_stay_on_the_circle(arith, gamma):
    """Products of two factors of modulus 1 within 2 u (and 2^-54 left of the
    correction), three roundings."""
    re, im = _table(gamma, 0.5, 255, arith)
    r = np.sqrt(re.astype(L) ** 2 + im.astype(L) ** 2)
    assert float(np.max(np.abs(r - L(0.5)))) <= 10 * 2.0 ** -53
