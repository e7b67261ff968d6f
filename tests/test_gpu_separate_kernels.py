"""The J-update's separate statistics kernels (csrc/ss.cu, ss_hessvec.cu, lm.cu) at one to three directions. Small
problems run as one launch by themselves (csrc/jupdate.cu); an explicit ctas_per_sm fixes the split of the
statistics sweeps and so takes the kernels that have one."""
import numpy as np
import pytest

from oracle import admm as O
from oracle import rtr as R
from paper_1502_00858_gb300 import Calibrator, capi
from synth import make_problem, user_layout

pytestmark = pytest.mark.gpu

N_LM, N_CG = 4, 3
SOLVERS = {"lm": capi.CALIB_JUPDATE_LM, "rtr": capi.CALIB_JUPDATE_RTR}


def c64(x):
    return np.asarray(x).astype(np.complex64).astype(np.complex128)


def _problem(N, K):
    """Two intervals, uneven samples, flagged baselines; the basis amplifies J into Z by less than 10."""
    return make_problem("adjoint_n16_k3", seed=61, N=N, K=K, P=5, I=2, T=(3, 5, 7), flag_max=0.2)


def _calibrator(prob, solver, **kw):
    cal = Calibrator(prob["N"], prob["pq"], prob["K"], prob["freqs"], prob["basis"], prob["rho"], n_intervals=prob["I"],
                     samples=prob["T"], n_lm=N_LM, n_cg=N_CG, jupdate=SOLVERS[solver], **kw)
    ul = user_layout(prob)
    cal.set_data(ul["vis"], ul["coh"], ul["flags"])
    return cal


@pytest.mark.parametrize("solver", sorted(SOLVERS))
def test_an_explicit_split_takes_the_kernels_that_have_one(lib, solver):
    """Launches of one iteration: statistics, residual sweep, evaluation, per step n_cg sweeps and CG steps, trial pass
    and evaluation, then gauge, fusion centre and records."""
    cal = _calibrator(_problem(13, 3), solver, ctas_per_sm=2)
    before = capi.calib_launch_count(cal.ctx)
    cal.iterate(1)
    assert capi.calib_launch_count(cal.ctx) - before == 3 + N_LM * (2 * N_CG + 2) + 3
    cal.close()


@pytest.mark.parametrize("solver", sorted(SOLVERS))
@pytest.mark.parametrize("N,K,m", [(8, 1, 1), (13, 3, 2), (34, 2, 1), (35, 1, 3), (41, 3, 1)])
def test_history_matches_the_oracle(lib, N, K, m, solver):
    """Tolerances as in the other C-ADMM histories (tests/test_gpu_parity.py): 1e-4 on objective and residual norm,
    1e-3 on primal and dual, the dual with an absolute floor of 1e-5 of its first record."""
    prob = _problem(N, K)
    cal = _calibrator(prob, solver, ctas_per_sm=m)
    hist = cal.iterate(3)
    cal.close()
    pr = dict(prob, V=[c64(v) for v in prob["V"]], C=[c64(c) for c in prob["C"]])
    kw = dict(n_lm=N_LM, n_cg=N_CG) if solver == "lm" else dict(
        jupdate=lambda J, V, C, pq, Y, BZ, rho: R.rtr_jupdate(J, V, C, pq, Y, BZ, rho, N_LM, N_CG))
    ref = O.admm(pr, 3, **kw)["hist"]
    amp = np.linalg.norm(np.linalg.pinv(prob["basis"].T @ prob["basis"]) @ prob["basis"].T, 2)
    assert amp < 10
    for key, rtol in (("objective", 1e-4), ("resid_norm", 1e-4), ("primal", 1e-3), ("dual", 1e-3)):
        np.testing.assert_allclose(hist[key], ref[key], rtol=rtol, atol=1e-5 * ref["dual"][0] if key == "dual" else 1e-7, err_msg=key)


@pytest.mark.parametrize("N,K", [(8, 1), (13, 3), (34, 2)])
def test_dependent_launch_changes_no_result(lib, N, K):
    """With profiling on the graph runs its kernels strictly one after another, else under programmatic dependent launch."""
    prob, out = _problem(N, K), []
    for profiling in (False, True):
        cal = _calibrator(prob, "lm", ctas_per_sm=2)
        capi.calib_profile_enable(cal.ctx, profiling)
        hist = cal.iterate(4)
        out.append([*hist.values(), *cal.solutions()])
        cal.close()
    for u, v in zip(*out):
        assert np.array_equal(u.view(np.uint8), v.view(np.uint8))


@pytest.mark.parametrize("solver", sorted(SOLVERS))
@pytest.mark.parametrize("N,K", [(8, 1), (13, 3), (34, 2), (41, 3)])
def test_one_launch_gives_the_bits_of_the_separate_kernels(lib, N, K, solver):
    """With one diagonal per piece (ctas_per_sm = 24: at most 200 diagonals here) the sums run in the same order: J, Z and
    Y after three iterations are the same bits, and the records, whose float64 sums are grouped differently, agree to 1e-12."""
    prob, out = _problem(N, K), []
    for m in (0, 24):
        cal = _calibrator(prob, solver, ctas_per_sm=m)
        before = capi.calib_launch_count(cal.ctx)
        hist = cal.iterate(3)
        out.append((capi.calib_launch_count(cal.ctx) - before, hist, cal.solutions()))
        cal.close()
    assert out[0][0] < out[1][0]
    for u, v in zip(out[0][2], out[1][2]):
        assert np.array_equal(u.view(np.uint8), v.view(np.uint8))
    for key in out[0][1]:
        np.testing.assert_allclose(out[0][1][key], out[1][1][key], rtol=1e-12, err_msg=key)
