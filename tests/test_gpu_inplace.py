"""calib_eval and calib_hessvec on device arrays: used where they are when 16-byte aligned and apart, through
the context's buffers otherwise. Every form gives the bits of the host-array call: aligned, 8-byte aligned,
the output in place of an input, and an output that overlaps its input in part."""
import numpy as np
import pytest

from paper_1502_00858_gb300 import Calibrator, capi
from synth import make_problem, user_layout

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", ["aligned", "offset", "alias", "overlap"])
@pytest.mark.parametrize("K", [1, 3])
def test_device_arrays_give_the_bits_of_host_arrays(lib, form, K):
    import torch

    prob = make_problem("adjoint_n16_k3", K=K)
    ul = user_layout(prob)
    cal = Calibrator(prob["N"], prob["pq"], K, prob["freqs"], prob["basis"], prob["rho"], samples=prob["T"])
    cal.set_data(ul["vis"], ul["coh"])
    rng = np.random.default_rng(3)
    J, eta = ((rng.standard_normal(cal.jones_shape + (2,)) * 0.3 + 0.5).astype(np.float32).view(np.complex64)[..., 0] for _ in range(2))
    L, g, grad = cal.eval(J)
    hv = cal.hessvec(J, eta)
    n = J.size * 2
    start = 2 if form == "offset" else 0
    pool = torch.zeros(6 * n, dtype=torch.float32, device="cuda")

    def place(x, at):
        pool[at:at + n] = torch.from_numpy(np.ascontiguousarray(x).view(np.float32).ravel()).cuda()
        return pool[at:at + n]

    def target(x, at):
        return x if form == "alias" else pool[at + 4:at + 4 + n] if form == "overlap" else pool[3 * n + start:4 * n + start]

    def check(t, want):
        capi.calib_sync(cal.ctx)
        np.testing.assert_array_equal(t.cpu().numpy(), np.ascontiguousarray(want).view(np.float32).ravel())

    Jd = place(J, start)
    out = target(Jd, start)
    Ld, gd = (torch.zeros(prob["A"], dtype=torch.float64, device="cuda") for _ in range(2))
    torch.cuda.synchronize()
    capi.calib_eval(cal.ctx, Jd, Ld, gd, out)
    check(out, grad)
    np.testing.assert_array_equal(gd.cpu().numpy(), g)
    np.testing.assert_array_equal(Ld.cpu().numpy(), L)

    Jd, Ed = place(J, 4 * n + start), place(eta, start)
    out = target(Ed, start)
    torch.cuda.synchronize()
    capi.calib_hessvec(cal.ctx, Jd, Ed, out)
    check(out, hv)
    cal.close()
