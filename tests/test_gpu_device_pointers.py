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


@pytest.mark.parametrize("correct", [-1, 1])
@pytest.mark.parametrize("offset", [0, 1, 3])
def test_residual_and_coherencies_into_any_complex_array(lib, offset, correct):
    """Outputs that start `offset` complex numbers (8 bytes each) into an allocation: the bits of the host-array calls,
    flagged baselines zeroed, and nothing around the outputs is touched."""
    import torch

    prob = make_problem("adjoint_n16_k3", N=13, K=3, P=5, I=2, T=(3, 5, 7), flag_max=0.25, seed=5)
    cal = _calibrator(prob)
    cal.set_initial(prob["J_true"].astype(np.complex64))
    sub = np.array([1, 0, 1], dtype=np.int32)
    res, coh = cal.residual(sub, None if correct < 0 else correct), cal.coherencies()
    for want, call in ((res, lambda out: capi.calib_residual(cal.ctx, out, sub, correct)),
                       (coh, lambda out: capi.calib_get_coherencies(cal.ctx, out))):
        buf = torch.full((want.size + 4,), 7.0, dtype=torch.complex64, device="cuda")
        torch.cuda.synchronize()
        call(buf[offset:offset + want.size])
        capi.calib_sync(cal.ctx)
        got = buf.cpu().numpy()
        np.testing.assert_array_equal(got[offset:offset + want.size].view(np.uint32), want.view(np.uint32))
        assert np.all(got[:offset] == 7) and np.all(got[offset + want.size:] == 7)
    cal.close()
