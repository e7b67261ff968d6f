"""Coherency prediction at the edges of its tiles: station counts that are no multiple of the 4-station blocks, the
smallest and the largest, source counts that leave a ragged last chunk, several groups of directions, and
uneven samples with flags, every element against the float64 oracle."""
import numpy as np
import pytest

from oracle import admm as O
from paper_1502_00858_gb300 import Calibrator, capi
from synth import make_problem, user_layout

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K,S,T,flagged", [(2, 1, 1, 1, 0.0), (3, 2, 3, (1, 3), 0.0), (5, 4, 7, 2, 0.2), (33, 3, 37, (1, 2), 0.1),
                                             (62, 5, 100, 1, 0.0), (63, 11, 19, (2, 1), 0.1), (101, 2, 130, 1, 0.0), (128, 3, 5, 1, 0.0)])
def test_predict_matches_oracle_at_tile_edges(lib, N, K, S, T, flagged):
    prob = make_problem("tiny_n8_k1", seed=97, N=N, K=K, P=4, I=1, T=T, flag_max=flagged)
    rng, ul = np.random.default_rng(97), user_layout(prob)
    sky = np.stack([rng.uniform(-0.05, 0.05, (K, S)), rng.uniform(-0.05, 0.05, (K, S)), rng.uniform(1.0, 10.0, (K, S)),
                    rng.uniform(-1.0, 1.0, (K, S))], axis=-1)
    cal = Calibrator(prob["N"], prob["pq"], prob["K"], prob["freqs"], prob["basis"], prob["rho"],
                     n_intervals=prob["I"], samples=prob["T"], formulation=capi.CALIB_FORM_DIRECT)
    cal.set_data(ul["vis"], ul["coh"], ul["flags"] if ul["flags"].any() else None)
    cal.predict(prob["uvw"], sky, prob["f0"])
    got, off = cal.coherencies(), 0
    for a in range(prob["A"]):
        iv, f = divmod(a, prob["P"])
        Ta = int(prob["T"][a])
        n = prob["B"] * Ta * K
        blk = got[off:off + n].reshape(prob["B"], Ta, K)
        off += n
        ref = O.predict_coherencies(prob["uvw"][iv, :Ta], sky, prob["freqs"][f], prob["f0"], prob["pq"])
        flux = (sky[..., 2] * (prob["freqs"][f] / prob["f0"]) ** sky[..., 3]).sum(-1)
        keep = prob["flags"][a] == 0
        # a source's term is off by a few float32 ulps of its flux, a chain of S sums by at most S half ulps of the
        # summed flux (130 * 2^-24 = 8e-6)
        assert np.all(np.abs(blk[keep] - ref[keep]) <= 2e-5 * flux)
        assert np.all(blk[~keep] == 0)
    cal.close()
