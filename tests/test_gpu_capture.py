"""Calls on device arrays recorded into a caller's CUDA graph: the graph stays good whatever the context does later."""
import numpy as np
import pytest

from paper_1502_00858_gb300 import Calibrator, capi
from synth import make_problem, user_layout

pytestmark = pytest.mark.gpu


def test_captured_prediction_survives_a_larger_one(lib):
    """A prediction is captured when the context already keeps a table of sources, a later one outside the graph
    needs a larger table, then the graph is replayed: it uses no memory that the context replaced (one kernel in
    the graph, which forms the sources itself) and gives the coherencies of the plain call, to the float32 rounding
    of the S-term sums (S 2^-24 of the flux)."""
    import torch

    prob = make_problem("adjoint_n16_k3")
    S = prob["sky"].shape[1]
    stream = torch.cuda.Stream()
    cal = Calibrator(prob["N"], prob["pq"], prob["K"], prob["freqs"], prob["basis"], prob["rho"], n_intervals=prob["I"],
                     samples=prob["T"], cuda_stream=stream.cuda_stream)
    cal.set_data(user_layout(prob)["vis"])
    uvw, sky = (torch.from_numpy(np.ascontiguousarray(prob[k], dtype=np.float64)).cuda() for k in ("uvw", "sky"))
    more = torch.cat([sky] * 40, dim=1).contiguous()
    torch.cuda.synchronize()
    cal.predict(uvw, sky, prob["f0"])
    want = cal.coherencies()
    graph = torch.cuda.CUDAGraph()
    before = capi.calib_launch_count(cal.ctx)
    with torch.cuda.graph(graph, stream=stream):
        cal.predict(uvw, sky, prob["f0"])
    assert capi.calib_launch_count(cal.ctx) - before == 1
    cal.predict(uvw, more, prob["f0"])
    capi.calib_sync(cal.ctx)
    assert np.abs(cal.coherencies() - want).max() > 0.1 * np.abs(want).max()
    with torch.cuda.stream(stream):
        graph.replay()
    torch.cuda.synchronize()
    flux = (prob["sky"][..., 2] * (prob["freqs"].max() / prob["f0"]) ** prob["sky"][..., 3]).sum(-1).max()
    assert np.abs(cal.coherencies() - want).max() <= S * 2.0 ** -24 * flux
    cal.close()
