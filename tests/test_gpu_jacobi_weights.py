"""The Jacobi weights of the LM preconditioner follow the coherencies: the statistics pass writes them when the
coherencies are new and leaves them alone when only the visibilities are. Whatever came before, a context iterates to
the bits of a new one that was given the same data."""
import numpy as np
import pytest

from paper_1502_00858_gb300 import Calibrator, capi
from synth import make_problem, user_layout

pytestmark = pytest.mark.gpu

N, K = 13, 4  # four directions: the separate kernels, which read the weights from global memory


def _problem(seed):
    return make_problem("adjoint_n16_k3", seed=seed, N=N, K=K, P=5, I=2, T=(3, 5, 7), flag_max=0.2)


def _calibrator(prob, **kw):
    return Calibrator(N, prob["pq"], K, prob["freqs"], prob["basis"], prob["rho"], n_intervals=prob["I"], samples=prob["T"],
                      n_lm=3, ctas_per_sm=2, **kw)


def _same(cal, vis, coh, flags):
    """cal from cold and a new context with the same arrays."""
    cal.reset()
    cal.iterate(2)
    new = _calibrator(_problem(91), formulation=cal.form)
    new.set_data(vis, coh, flags)
    new.iterate(2)
    for u, v in zip(cal.solutions(), new.solutions()):
        assert np.array_equal(u.view(np.uint8), v.view(np.uint8))
    new.close()


@pytest.mark.parametrize("form", [capi.CALIB_FORM_STATISTICS, capi.CALIB_FORM_DIRECT])
def test_weights_follow_the_coherencies(lib, form):
    a, b = user_layout(_problem(91)), user_layout(_problem(92))
    cal = _calibrator(_problem(91), formulation=form)
    cal.form = form
    cal.set_data(a["vis"], a["coh"], a["flags"])
    _same(cal, a["vis"], a["coh"], a["flags"])
    cal.set_data(b["vis"])  # visibilities alone
    _same(cal, b["vis"], a["coh"], a["flags"])
    cal.set_data(b["vis"], b["coh"])  # new coherencies
    _same(cal, b["vis"], b["coh"], a["flags"])
    cal.set_data(a["vis"], a["coh"], b["flags"])  # another layout
    cal.set_data(b["vis"])
    _same(cal, b["vis"], a["coh"], b["flags"])
    prob = _problem(91)
    cal.predict(prob["uvw"], prob["sky"], prob["f0"])
    cal.set_data(a["vis"])
    _same(cal, a["vis"], cal.coherencies(), b["flags"])
    cal.close()


def test_weights_follow_coherencies_that_a_graph_writes(lib):
    """A recorded prediction changes the coherencies at every replay, without a call."""
    import torch

    prob, a = _problem(91), user_layout(_problem(91))
    stream = torch.cuda.Stream()
    cal = _calibrator(prob, cuda_stream=stream.cuda_stream)
    cal.form = capi.CALIB_FORM_STATISTICS
    cal.set_data(a["vis"], a["coh"], a["flags"])
    uvw, sky = (torch.from_numpy(np.ascontiguousarray(prob[k], dtype=np.float64)).cuda() for k in ("uvw", "sky"))
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        cal.predict(uvw, sky, prob["f0"])
    _same(cal, a["vis"], a["coh"], a["flags"])
    sky[..., 2] *= 3.0
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        graph.replay()
    torch.cuda.synchronize()
    cal.set_data(a["vis"])
    coh = cal.coherencies()
    assert np.abs(coh - np.where(coh == 0, 0, a["coh"])).max() > 0.1 * np.abs(a["coh"]).max()
    _same(cal, a["vis"], coh, a["flags"])
    cal.close()
