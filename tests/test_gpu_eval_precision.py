"""calib_eval returns L in float64 and forms its penalty part, Re tr(Y^H D) + rho/2 ||D||^2 with D = J - BZ, in float64 as
well. Without visibilities and coherencies (all zero) g is exactly 0, and L is the penalty alone."""
from fractions import Fraction

import numpy as np
import pytest

from paper_1502_00858_gb300 import Calibrator, capi

pytestmark = pytest.mark.gpu

N, P = 2, 64
PQ = np.array([[0, 1]], dtype=np.int32)


def _calibrator(rho):
    """One direction, a constant basis: B_i Z is Z itself, exact for a float32 Z."""
    cal = Calibrator(N, PQ, 1, np.linspace(100e6, 200e6, P), np.ones((P, 1)), [rho])
    cal.set_data(np.zeros(P * 4, dtype=np.complex64), np.zeros(P, dtype=np.complex64))
    return cal


def test_penalty_has_float64_precision(lib):
    """Each agent has one number with J != BZ, and there Y cancels rho/2 D to the rounding of Y. The exact value is
    d (y + h d) with h = rho/2 (fractions); d is exact in float64, the inner sum is a product of at most
    62 bits and y, each rounded by at most 2^-53 of h d, and the last product by 2^-53 of a far smaller one: the
    error is at most 2^-52 |d| |h d|."""
    rng = np.random.default_rng(71)
    rho = float(np.float32(5.3))
    cal = _calibrator(rho)
    bz = np.float32(rng.uniform(1e-4, 2e-4))
    Z = np.zeros((1, 1, 1, N, 2, 2), dtype=np.complex128)
    Z[0, 0, 0, 0, 0, 0] = float(bz)
    J = np.zeros((P, 1, N, 2, 2), dtype=np.complex64)
    Y = np.zeros_like(J)
    j = rng.uniform(0.5, 1.5, P).astype(np.float32)
    d = j.astype(np.float64) - float(bz)
    y = (-0.5 * rho * d).astype(np.float32)
    J[:, 0, 0, 0, 0], Y[:, 0, 0, 0, 0] = j, y
    cal.set_consensus(Z, Y)
    L, g, grad = cal.eval(J)
    cal.close()
    assert np.all(g == 0)
    for a in range(P):
        D = Fraction(float(j[a])) - Fraction(float(bz))
        hd = Fraction(rho) / 2 * D
        want = D * (Fraction(float(y[a])) + hd)
        assert abs(Fraction(float(L[a])) - want) <= abs(D * hd) / 2 ** 52, a
        want_grad = float(Fraction(float(y[a])) / 2 + hd)
        assert grad[a, 0, 0, 0, 0].real == pytest.approx(want_grad, rel=2.0 ** -23, abs=0)


@pytest.mark.parametrize("size", [1e-21, 1e-10, 1e15, 1e20, 1e30])
def test_penalty_has_float64_range(lib, size):
    """Entries whose squares leave float32: the penalty rho/2 |J|^2 of 16 equal entries to 16 rounding errors of 2^-53."""
    rho = 5.0
    cal = _calibrator(rho)
    cal.set_consensus(None, None)
    x = np.float32(size)
    J = np.zeros((P, 1, N, 2, 2), dtype=np.complex64)
    J[:, 0, 0] = x
    L, g, grad = cal.eval(J)
    cal.close()
    np.testing.assert_allclose(L - g, 4 * 0.5 * rho * float(x) ** 2, rtol=2.0 ** -48)
    np.testing.assert_allclose(grad[:, 0, 0].real, 0.5 * rho * float(x), rtol=2.0 ** -23)
