"""The J-update in one launch (small problems, csrc/jupdate.cu) at the edges of its range: the smallest
network, odd station counts, sums taken in several chunks of diagonals, more agents than SMs (the smaller
CTA), every direction count, both inner solvers. The first J-update from the cold start is independent of the
other agents, so the data cost it reaches is compared agent by agent with the oracle's J-update on the same
inputs, at the 1e-4 of the other C-ADMM comparisons (float32 passes; a wrong station sum or a missed slot
changes the step and with it the cost far more)."""
import numpy as np
import pytest

from oracle import admm as O
from oracle import rtr as R
from paper_1502_00858_gb300 import Calibrator, capi
from synth import make_problem, user_layout

pytestmark = pytest.mark.gpu

# N, K, P, I, flagged share, solver
SHAPES = [
    (2, 1, 3, 1, 0.0, "lm"),
    (3, 3, 4, 1, 0.0, "rtr"),
    (16, 3, 4, 45, 0.1, "lm"),    # 180 agents
    (33, 1, 3, 1, 0.2, "lm"),
    (33, 2, 3, 60, 0.0, "rtr"),   # 180 agents
    (47, 3, 3, 1, 0.05, "lm"),    # the sums take several chunks of diagonals
    (62, 2, 4, 1, 0.0, "lm"),
    (64, 1, 3, 1, 0.0, "rtr"),
]


def c64(x):
    return np.asarray(x).astype(np.complex64).astype(np.complex128)


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: f"n{s[0]}_k{s[1]}_a{s[2] * s[3]}_{s[5]}")
def test_first_jupdate_matches_the_oracle(lib, shape):
    N, K, P, I, flagged, solver = shape
    prob = make_problem("tiny_n8_k1", seed=31, N=N, K=K, P=P, I=I, T=3, flag_max=flagged)
    ul = user_layout(prob)
    cal = Calibrator(N, prob["pq"], K, prob["freqs"], prob["basis"], prob["rho"], n_intervals=I, samples=prob["T"],
                     n_lm=4, n_cg=3, jupdate=capi.CALIB_JUPDATE_LM if solver == "lm" else capi.CALIB_JUPDATE_RTR)
    cal.set_data(ul["vis"], ul["coh"], ul["flags"] if ul["flags"].any() else None)
    before = capi.calib_launch_count(cal.ctx)
    cal.iterate(1)
    # statistics, residual sweep, J-update, gauge, fusion centre, records (9 launches a step otherwise)
    assert capi.calib_launch_count(cal.ctx) - before == 6
    _, g = cal.agent_objective()
    cal.close()
    step = O.lm_jupdate if solver == "lm" else R.rtr_jupdate
    for a in sorted({0, P - 1, P * I - 1}):
        keep = prob["flags"][a] == 0
        V, C, pq = c64(prob["V"][a][keep]), c64(prob["C"][a][keep]), prob["pq"][keep]
        J0 = np.broadcast_to(np.eye(2, dtype=complex), (K, N, 2, 2)).copy()
        zero = np.zeros_like(J0)
        J = step(J0, V, C, pq, zero, zero, prob["rho"], 4, 3)
        assert g[a] == pytest.approx(O.data_cost(J, V, C, pq), rel=1e-4), a
