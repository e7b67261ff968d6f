"""The autotuner's results are shared between contexts of one shape in a process, but only where the candidates are timed
as the context's solver launches them."""
import pytest

from paper_1502_00858_gb300 import Calibrator, capi
from synth import make_problem, user_layout

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", [capi.CALIB_FORM_STATISTICS, capi.CALIB_FORM_DIRECT])
def test_a_solver_does_not_take_another_ones_split(lib, form):
    """Launches of the first iteration, which include the autotuner's: the LM context tunes although a trust-region one
    of its shape has; a second LM context does not, nor does a second trust-region one."""
    prob = make_problem("adjoint_n16_k3", N=14, K=4, P=4, I=1, T=2, seed=67)
    ul = user_layout(prob)

    def launches(solver):
        cal = Calibrator(prob["N"], prob["pq"], prob["K"], prob["freqs"], prob["basis"], prob["rho"],
                         samples=prob["T"], n_lm=2, n_cg=3, formulation=form, jupdate=solver)
        cal.set_data(ul["vis"], ul["coh"])
        before = capi.calib_launch_count(cal.ctx)
        cal.iterate(1)
        n = capi.calib_launch_count(cal.ctx) - before
        cal.close()
        return n

    rtr, lm = capi.CALIB_JUPDATE_RTR, capi.CALIB_JUPDATE_LM
    first = [launches(s) for s in (rtr, lm)]
    again = [launches(s) for s in (rtr, lm)]
    assert first[0] > again[0] and first[1] > again[1], (first, again)
