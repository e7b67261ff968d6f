"""Data in and out of the internal layout: bit-exact round trips of visibilities (a residual that subtracts
nothing) and coherencies, at station counts with and without padded slots, several CTA passes a diagonal,
reversed pairs, ragged samples and flags; a source that is only 8-byte aligned; the non-finite check, which also
covers flagged baselines."""
import numpy as np
import pytest

from paper_1502_00858_gb300 import Calibrator, capi
from synth import make_problem, user_layout

pytestmark = pytest.mark.gpu


def _problem(N, K, T, flagged):
    return make_problem("tiny_n8_k1", seed=41, N=N, K=K, P=4, I=1, T=T, flag_max=flagged)


def _calibrator(prob):
    return Calibrator(prob["N"], prob["pq"], prob["K"], prob["freqs"], prob["basis"], prob["rho"],
                      n_intervals=prob["I"], samples=prob["T"])


def _expected(flat, prob, w):
    """The user-layout array with its flagged baselines zeroed."""
    out, off = flat.copy(), 0
    for a in range(prob["A"]):
        n = prob["B"] * int(prob["T"][a]) * w
        block = out[off:off + n].reshape(prob["B"], -1)
        block[prob["flags"][a] != 0] = 0
        off += n
    return out


@pytest.mark.parametrize("N,K,T,flagged", [(2, 1, 1, 0.0), (7, 2, (1, 4, 6), 0.3), (62, 5, 3, 0.1), (70, 3, (2, 5), 0.2),
                                           (128, 1, 2, 0.0)])
@pytest.mark.parametrize("offset", [0, 1])
def test_round_trip_is_exact(lib, N, K, T, flagged, offset):
    import torch

    prob = _problem(N, K, T, flagged)
    ul = user_layout(prob)

    def device(x):  # starts `offset` complex numbers (8 bytes each) into its allocation
        base = torch.zeros((x.size + offset) * 2, dtype=torch.float32, device="cuda")
        base[2 * offset:] = torch.from_numpy(x.view(np.float32)).cuda()
        return base[2 * offset:]

    cal = _calibrator(prob)
    torch.cuda.synchronize()
    vis, coh = device(ul["vis"]), device(ul["coh"])
    flags = torch.from_numpy(ul["flags"]).cuda() if ul["flags"].any() else None
    torch.cuda.synchronize()
    cal.set_data(vis, coh, flags)
    out = cal.residual(subtract=np.zeros(K, dtype=np.int32))
    np.testing.assert_array_equal(out, _expected(ul["vis"], prob, 4))
    np.testing.assert_array_equal(cal.coherencies(), _expected(ul["coh"], prob, K))
    cal.close()


@pytest.mark.parametrize("what", ["vis", "coh"])
@pytest.mark.parametrize("flagged_one", [True, False])
def test_non_finite_values_are_found_everywhere(lib, what, flagged_one):
    prob = _problem(9, 2, 3, 0.3)
    ul = user_layout(prob)
    a, b = next((a, b) for a in range(prob["A"]) for b in range(prob["B"]) if bool(prob["flags"][a][b]) == flagged_one)
    w = 4 if what == "vis" else prob["K"]
    ul[what][((a * prob["B"]) + b + 1) * 3 * w - 1] = np.nan + 0j  # the last value of that baseline
    cal = _calibrator(prob)
    with pytest.raises(capi.CalibError) as err:
        cal.set_data(ul["vis"], ul["coh"], ul["flags"])
    assert err.value.code == capi.CALIB_ENUMERIC
    cal.close()
