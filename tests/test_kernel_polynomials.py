"""The double plans' per-tap polynomials as the host fits them (no GPU): which
kernel shapes take them, and how far they are from the kernel's definition."""
import ctypes

import numpy as np
import pytest
from scipy.special import ive

from paper_1502_05037_gb300 import _lib, build as pbuild

MAX_J, MAX_DEG = 8, 18


class KbPolyD(ctypes.Structure):
    _fields_ = [("J", ctypes.c_int), ("poly", ctypes.c_int), ("beta", ctypes.c_double), ("inv_i0beta", ctypes.c_double),
                ("coef", (ctypes.c_double * (MAX_DEG + 1)) * MAX_J)]


@pytest.fixture(scope="module")
def fit():
    pbuild.build()
    f = getattr(_lib.load(), "_ZN6purify13fit_kb_poly_dEid")   # purify::fit_kb_poly_d(int, double)
    f.restype, f.argtypes = KbPolyD, [ctypes.c_int, ctypes.c_double]
    return f


def tap(J, a, beta, z):
    t = 0.5 * z + (0.5 * J - 0.5 - a)
    s = np.sqrt(np.maximum(1.0 - (2.0 * t / J) ** 2, 0.0))
    return ive(0, beta * s) / ive(0, beta) * np.exp(beta * (s - 1.0))


@pytest.mark.parametrize("J", range(2, 9))
def test_default_shape_is_a_polynomial(fit, J):
    kp = fit(J, 2.34 * J)
    assert (kp.J, kp.poly, kp.beta) == (J, 1, 2.34 * J)
    again = fit(J, 2.34 * J)
    z = np.linspace(-1.0, 1.0, 801)
    for a in range(J):
        c = np.array(kp.coef[a])
        assert np.array_equal(c, np.array(again.coef[a]))
        # the definition in doubles: scipy's i0e to a few units, an exponential
        # of up to beta units more
        assert np.abs(np.polyval(c[::-1], z) - tap(J, a, kp.beta, z)).max() <= (4 + kp.beta) * 2.3e-16


@pytest.mark.parametrize("J", range(2, 9))
def test_wide_shapes_keep_the_definition(fit, J):
    assert fit(J, 5.0 * J).poly == 0
    assert fit(J, 1.0 * J).poly == 1     # narrower than the default: a lower degree would do
