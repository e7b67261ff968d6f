"""Which problems run their J-update as one launch: only those that it was measured to be the faster form of, on both
sides of the rule's limits. Where it does run, it gives the bits of the separate kernels with one diagonal per piece."""
import numpy as np
import pytest

from paper_1502_00858_gb300 import Calibrator, capi

pytestmark = pytest.mark.gpu

N_LM, N_CG = 2, 3
# N, K, agents per SM of 152 (A / 152 rounded up to whole intervals of four subbands), solver, one launch
RULE = [
    (80, 1, 16, "lm", True), (96, 1, 16, "lm", False), (96, 1, 16, "rtr", False), (128, 1, 80, "lm", True), (128, 1, 80, "rtr", False),
    (63, 2, 16, "lm", True), (63, 2, 16, "rtr", False), (47, 3, 16, "lm", True), (47, 3, 16, "rtr", False), (47, 3, 80, "rtr", True),
    (80, 1, 160, "lm", True), (84, 1, 160, "lm", False), (64, 1, 160, "rtr", True), (80, 1, 160, "rtr", False), (34, 3, 160, "rtr", True),
    (88, 1, 320, "lm", False), (28, 1, 640, "lm", True), (28, 1, 640, "rtr", False), (20, 2, 640, "lm", True), (16, 1, 640, "rtr", False),
    (16, 1, 600, "rtr", True), (20, 1, 2560, "lm", False), (33, 1, 2560, "lm", True), (20, 2, 2560, "lm", False), (10, 2, 2560, "rtr", True),
    (12, 1, 2560, "rtr", False),
]


def _run(N, K, A, solver, m):
    P, rng = 4, np.random.default_rng(83)
    pq = np.stack(np.triu_indices(N, 1), 1).astype(np.int32)
    freqs = np.linspace(120e6, 160e6, P)
    cal = Calibrator(N, pq, K, freqs, np.ones((P, 1)), np.full(K, 5.0), n_intervals=A // P, n_lm=N_LM, n_cg=N_CG, ctas_per_sm=m,
                     jupdate=capi.CALIB_JUPDATE_LM if solver == "lm" else capi.CALIB_JUPDATE_RTR)
    cn = lambda *s: rng.standard_normal((*s, 2), dtype=np.float32).view(np.complex64)[..., 0]  # noqa: E731
    coh = cn(A, len(pq), K)
    vis = np.float32(0.1) * cn(A, len(pq), 2, 2)
    s = coh.sum(-1)
    vis[..., 0, 0] += np.float32(1.1) * s
    vis[..., 1, 1] += np.float32(0.9) * s
    cal.set_data(vis, coh)
    if m == 0:  # warm the autotuner of the separate kernels: its launches are not the iteration's
        cal.iterate(1)
        cal.reset()
    before = capi.calib_launch_count(cal.ctx)
    cal.iterate(1)
    n = capi.calib_launch_count(cal.ctx) - before
    out = cal.solutions()
    cal.close()
    return n, out


@pytest.mark.parametrize("N,K,A,solver,one", RULE)
def test_one_launch_only_where_it_is_faster(lib, N, K, A, solver, one):
    import torch

    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the agents of the table are meant for 152 SMs")
    n, out = _run(N, K, A, solver, 0)
    # residual sweep, J-update, gauge, fusion centre, records; or its evaluation and its steps' kernels
    assert n == (5 if one else 5 + N_LM * (2 * N_CG + 2))
    if one and A <= 160:
        _, ref = _run(N, K, A, solver, (A * (N // 2) + 151) // 152)
        for u, v in zip(out, ref):
            assert np.array_equal(u.view(np.uint8), v.view(np.uint8))
