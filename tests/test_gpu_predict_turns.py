"""The fraction of the turns in the prediction, at its edges: whole and half turns of both signs, which float32 phasors
hold exactly, and turns on both sides of 2^-12, where the way that the fraction is cut out changes."""
import numpy as np
import pytest

from paper_1502_00858_gb300 import Calibrator

pytestmark = pytest.mark.gpu

C_LIGHT = 299792458.0


def test_fractions_of_turns(lib):
    """One source at l = 1/16, f / c = 1 and stations on the u axis: turns u / 16, all exact in float64. Quarter, half and
    whole turns give exact phasors, so the coherencies are exact; the others are within 4 float32 roundings of 1."""
    turns = np.array([0.0, 0.5, -0.5, 1.0, -1.0, 4096.5, -4096.5, 0.25, -0.25, 2.0 ** 40 + 0.5, -(2.0 ** 40 + 0.5), 2.0 ** 51 + 0.5,
                      2.0 ** 60, 2.0 ** -12, -2.0 ** -12, 2.0 ** -13, -2.0 ** -13, 3.0 + 2.0 ** -30, -1e-300])
    N = len(turns)
    pq = np.stack(np.triu_indices(N, 1), 1).astype(np.int32)
    cal = Calibrator(N, pq, 1, [C_LIGHT], [[1.0]], [5.0])
    uvw = np.zeros((1, 1, N, 3))
    uvw[0, 0, :, 0] = turns * 16
    cal.set_data(np.zeros(len(pq) * 4, dtype=np.complex64))
    cal.predict(uvw, np.array([[[0.0625, 0.0, 1.0, 0.0]]]), C_LIGHT)
    got = cal.coherencies()
    cal.close()
    frac = turns - np.rint(turns)
    exact = np.isin(np.abs(frac), (0.0, 0.25, 0.5))
    quarter = np.where(exact, np.round(4 * frac), 0).astype(int) % 4
    e = np.where(exact, np.array([1, -1j, -1, 1j])[quarter], np.exp(-2j * np.pi * frac))
    want = e[pq[:, 0]] * np.conj(e[pq[:, 1]])
    both = exact[pq[:, 0]] & exact[pq[:, 1]]
    np.testing.assert_array_equal(got[both], want[both].astype(np.complex64))
    assert np.abs(got - want).max() <= 4 * 2.0 ** -23
