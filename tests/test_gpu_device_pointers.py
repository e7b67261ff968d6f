"""Device arrays that are not aligned for the kernels' widest accesses: the call gives what it gives with aligned ones."""
import numpy as np
import pytest

from paper_1502_00858_gb300 import Calibrator, capi
from synth import make_problem, user_layout

pytestmark = pytest.mark.gpu


def _calibrator(prob):
    cal = Calibrator(prob["N"], prob["pq"], prob["K"], prob["freqs"], prob["basis"], prob["rho"],
                     n_intervals=prob["I"], samples=prob["T"])
    ul = user_layout(prob)
    cal.set_data(ul["vis"], ul["coh"], ul["flags"] if ul["flags"].any() else None)
    return cal


@pytest.mark.parametrize("off_L,off_g", [(4, 0), (0, 4), (4, 4), (8, 8)])
def test_eval_writes_scalars_to_any_address(lib, off_L, off_g):
    """L and g of calib_eval start off_L and off_g bytes past a 16-byte boundary: the bits of the host-array call,
    and nothing around them is touched."""
    import torch

    prob = make_problem("adjoint_n16_k3")
    cal = _calibrator(prob)
    J = prob["J_true"].astype(np.complex64)
    L, g, _ = cal.eval(J)
    n = prob["A"] * 8
    Jd = torch.from_numpy(J.view(np.float32)).cuda()
    grad = torch.empty_like(Jd)
    buf = [torch.full((n + 32,), 7, dtype=torch.uint8, device="cuda") for _ in range(2)]
    torch.cuda.synchronize()
    capi.calib_eval(cal.ctx, Jd, buf[0][off_L:off_L + n], buf[1][off_g:off_g + n], grad)
    capi.calib_sync(cal.ctx)
    for b, off, want in ((buf[0], off_L, L), (buf[1], off_g, g)):
        got = b.cpu().numpy()
        np.testing.assert_array_equal(got[off:off + n], want.view(np.uint8))
        assert np.all(got[:off] == 7) and np.all(got[off + n:] == 7)
    cal.close()
