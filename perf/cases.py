"""The calls that a user of this framework makes, at the sizes they are made at, for timing.

Each case is one use of a public entry point (the Calibrator context, the C names in capi, the autograd
loss, the warm-start network) on device arrays, as bench.py and the drivers of this package make them:

  calibrate   sky model and visibilities in, solutions out: predict, cold start, C-ADMM iterations
  track       the next solution interval: new visibilities in, start from the previous solution
              (refined by the network where `net` is set), a few iterations, solutions out
  gradient    L and grad L of every agent at a given J (an outside optimiser or an end-to-end loss)
  loss        the same through the differentiable loss, forward and backward
  hessian     a Gauss-Newton Hessian-vector product of every agent
  apply       new visibilities and coherencies in, the solutions subtracted and the data corrected
  predict     coherencies of the sky model out
  train       one optimiser step of the warm-start network

The synthetic inputs follow the observations that the framework is for (point-source clusters in a 7 degree
field seen by a LOFAR-like array, Jones matrices smooth in frequency, noise); they are formed here with torch.
Z and the objective are stored in float64 but rest on float32 solutions and residuals, so they are returned
in 32 bits, as a program that goes on with them beside J does.
"""
import math

import numpy as np
import torch

from paper_1502_00858_gb300 import Calibrator, capi
from paper_1502_00858_gb300.adjoint import admm_loss
from paper_1502_00858_gb300.warmstart import WarmStartNet, init_weights

C_LIGHT = 299792458.0
F0 = 150e6
JUPDATE = {"lm": capi.CALIB_JUPDATE_LM, "rtr": capi.CALIB_JUPDATE_RTR, "sage": capi.CALIB_JUPDATE_SAGE}


def _case(name, what, **kw):
    c = {"name": name, "what": what}
    c.update(kw)
    return c


def _shape(N, K, P, I, T, S=20, M=4, rho=10.0, Tmin=0, flagged=0.0):
    """N stations, K directions of S sources, P subbands x I solution intervals, T samples (ragged from Tmin up
    where that is set), M basis terms, share of flagged baselines."""
    return {"N": N, "K": K, "P": P, "I": I, "T": T, "Tmin": Tmin or T, "S": S, "M": M, "rho": rho, "flagged": flagged}


def listed():
    return [
        # the smallest network (8 stations, 4 subbands) calibrated from cold: launches and latency
        _case("calibrate n8 k1", "calibrate", iters=5, n_lm=10, n_cg=4, jupdate="lm", **_shape(8, 1, 4, 1, 10, S=4, M=3, rho=5.0)),
        # the paper's first simulation: one direction, 47 stations, 32 channels, one interval
        _case("calibrate n47 k1", "calibrate", iters=5, n_lm=10, n_cg=4, jupdate="lm", **_shape(47, 1, 32, 1, 20, S=1, M=2, rho=5.0)),
        # a third of the benchmark's workload (10 of its 30 iterations): 62 stations, 5 directions, 32 subbands x 10 intervals
        _case("calibrate n62 k5", "calibrate", iters=10, n_lm=10, n_cg=4, jupdate="lm", **_shape(62, 5, 32, 10, 10)),
        # the batched uneven survey: 10 directions, 256 subbands, 5 to 20 samples, flagged baselines
        _case("calibrate n62 k10 uneven", "calibrate", iters=3, n_lm=10, n_cg=4, jupdate="lm",
              **_shape(62, 10, 256, 4, 20, Tmin=5, flagged=0.08)),
        # the paper's own inner solver (trust region) at a mid-sized network
        _case("calibrate n30 k3 rtr", "calibrate", iters=3, n_lm=10, n_cg=4, jupdate="rtr", **_shape(30, 3, 16, 2, 7)),
        # a running observation: the next interval from the last one's solution, refined by the network
        _case("track n62 k5", "track", iters=2, n_lm=10, n_cg=4, jupdate="lm", net=True, **_shape(62, 5, 64, 1, 10)),
        # gradients for an outside optimiser over the whole batch
        _case("gradient n62 k5", "gradient", **_shape(62, 5, 32, 10, 10)),
        # the differentiable loss at the size of an end-to-end training check
        _case("loss n16 k3", "loss", **_shape(16, 3, 8, 1, 2, S=5)),
        # curvature for an outside second-order method: many directions, ragged samples
        _case("hessian n47 k10 ragged", "hessian", **_shape(47, 10, 64, 1, 20, Tmin=5, flagged=0.05)),
        # the pass over the data after calibration: subtract every direction, correct towards one
        _case("apply n62 k5", "apply", **_shape(62, 5, 32, 10, 10, flagged=0.05)),
        # a deep sky model: 100 sources a cluster
        _case("predict n62 k5 s100", "predict", **_shape(62, 5, 32, 2, 10, S=100)),
        # the warm-start network's optimiser step at its driver's batch
        _case("train w256", "train", width=256, depth=3, rows=2048),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    what = rng.choice(["calibrate", "calibrate", "track", "gradient", "loss", "hessian", "apply", "predict", "train"])
    if what == "train":
        return {"what": what, "width": rng.choice([64, 128, 200, 256]), "depth": rng.randint(1, 3), "rows": _log_int(rng, 300, 4096)}
    while True:
        K = _log_int(rng, 1, 10)
        c = {"what": what}
        c.update(_shape(_log_int(rng, 8, 62), K, _log_int(rng, 4, 256), rng.randint(1, 10), rng.randint(4, 20),
                        S=_log_int(rng, 1, 100 if what == "predict" else 20), M=rng.randint(2, 4),
                        flagged=rng.choice([0.0, 0.0, rng.uniform(0.01, 0.15)])))
        if what == "loss":
            c["P"], c["I"], c["flagged"] = _log_int(rng, 4, 32), 1, 0.0
        if what == "predict":
            c["flagged"] = 0.0
        if rng.random() < 0.4:
            c["Tmin"] = rng.randint(2, c["T"])
        if what in ("calibrate", "track"):
            c.update(iters=rng.randint(1, 3), n_lm=10, n_cg=4, jupdate="lm")
            if what == "calibrate" and rng.random() < 0.2:
                c["jupdate"], c["iters"] = "rtr", rng.randint(1, 2)
            if what == "track":
                c["net"] = rng.random() < 0.5
                c["flagged"] = 0.0
        w, top = work(c), work(listed()[3])
        if w["flops"] <= 0.5 * top["flops"] and w["bytes"] <= 0.5 * top["bytes"]:
            return c


# ----------------------------------------------------------------------------- inputs

class Obs:
    """One synthetic observation: the arrays of the problem, on the GPU where the calls take them there."""


def _pairs(N):
    i, j = np.triu_indices(N, 1)
    return np.stack([i, j], 1).astype(np.int32)


def _basis(freqs, M):
    """Bernstein polynomials over the band (an ordinary polynomial of degree 1 where M is 2)."""
    x = (freqs - freqs.min()) / max(freqs.max() - freqs.min(), 1.0)
    if M == 2:
        return np.stack([np.ones_like(freqs), (freqs - F0) / F0], 1)
    return np.stack([math.comb(M - 1, l) * x ** l * (1 - x) ** (M - 1 - l) for l in range(M)], 1)


def _coherencies(o, a0, a1, Ta, dtype):
    """c [a1-a0, B, Ta, K] of the agents a0..a1 of one interval, all with Ta samples (Eq. coh)."""
    iv = a0 // o.P
    f = o.freqs_t[[a % o.P for a in range(a0, a1)]]
    turns = torch.einsum("tnx,ksx->tnks", o.uvw[iv, :Ta], o.dirs)  # metres
    turns = (f / C_LIGHT)[:, None, None, None, None] * turns
    turns = turns - torch.round(turns)
    rdt = torch.float64 if dtype == torch.complex128 else torch.float32
    ph = (-2 * math.pi * turns).to(rdt)
    E = torch.polar(torch.ones_like(ph), ph).permute(0, 1, 3, 2, 4)  # [a, t, K, N, S]
    flux = (o.sky[:, :, 2] * (f[:, None, None] / F0) ** o.sky[:, :, 3]).to(rdt)  # [a, K, S]
    G = torch.matmul(E * flux[:, None, :, None, :], E.conj().transpose(-1, -2))
    return G[..., o.p, o.q].permute(0, 3, 1, 2)


def _groups(o):
    """Runs of consecutive agents of one interval with the same sample count, at most 64 (or less work) long."""
    a, out = 0, []
    most = max(1, min(64, int(4e8 / (o.Tmax * o.K * o.N * (o.N + o.S)) / 8)))
    while a < o.A:
        b = a + 1
        while b < o.A and b - a < most and o.T[b] == o.T[a] and b // o.P == a // o.P:
            b += 1
        out.append((a, b, int(o.T[a])))
        a = b
    return out


def _observation(case, seed, vis=True, coh=False):
    o = Obs()
    dev = torch.device("cuda")
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device=dev).manual_seed(seed)
    o.N, o.K, o.P, o.I, o.S, o.M = (case[k] for k in ("N", "K", "P", "I", "S", "M"))
    o.A = o.I * o.P
    o.pq = _pairs(o.N)
    o.B = len(o.pq)
    o.p, o.q = (torch.from_numpy(o.pq[:, i].astype(np.int64)).to(dev) for i in (0, 1))
    o.freqs = np.linspace(115e6, 185e6, o.P)
    o.freqs_t = torch.from_numpy(o.freqs).to(dev)
    o.M = min(o.M, o.P)
    o.basis = _basis(o.freqs, o.M)
    o.rho = np.full(o.K, float(case["rho"]))
    sub = np.sort(rng.integers(case["Tmin"], case["T"] + 1, o.P))  # samples of each subband
    sub[-1] = case["T"]
    o.T = np.tile(sub, o.I).astype(np.int32)
    o.Tmax = int(o.T.max())
    # stations out to 40 km, tracked at the north celestial pole, 10 s samples
    r, az = np.exp(rng.uniform(math.log(50.0), math.log(40e3), o.N)), rng.uniform(0, 2 * math.pi, o.N)
    e, n, u = r * np.sin(az), r * np.cos(az), rng.normal(0.0, 10.0, o.N)
    s, c = math.sin(math.radians(52.9)), math.cos(math.radians(52.9))
    X, Y, Z = -s * n + c * u, e, c * n + s * u
    H = 0.3 + 2 * math.pi / 86164.0905 * 10.0 * np.arange(o.I * o.Tmax)[:, None]
    uvw = np.stack([np.sin(H) * X + np.cos(H) * Y, -np.cos(H) * X + np.sin(H) * Y, np.broadcast_to(Z, (len(H), o.N))], -1)
    o.uvw = torch.from_numpy(uvw.reshape(o.I, o.Tmax, o.N, 3).copy()).to(dev)
    # clusters of half a degree inside a 7 degree field, Pareto fluxes, spectral indices U(-1, 1)
    half = math.radians(3.5)
    centre = rng.uniform(-half, half, (o.K, 2))
    rad, ang = math.radians(0.5) * np.sqrt(rng.uniform(0, 1, (o.K, o.S))), rng.uniform(0, 2 * math.pi, (o.K, o.S))
    sky = np.stack([np.sin(centre[:, :1] + rad * np.cos(ang)), np.sin(centre[:, 1:] + rad * np.sin(ang)),
                    1.0 + rng.pareto(1.5, (o.K, o.S)), rng.uniform(-1, 1, (o.K, o.S))], -1)
    # clusters of like total flux: none is lost beside the others
    sky[..., 2] *= (10.0 * rng.uniform(1.0, 2.0, (o.K, 1))) / sky[..., 2].sum(1, keepdims=True)
    o.sky = torch.from_numpy(sky).to(dev)
    lmn = np.stack([sky[..., 0], sky[..., 1], np.sqrt(1 - sky[..., 0] ** 2 - sky[..., 1] ** 2) - 1], -1)
    o.dirs = torch.from_numpy(lmn).to(dev)
    # identity plus a polynomial in frequency that drifts between the intervals, and a per-channel part
    cn = lambda *sh: (rng.standard_normal(sh) + 1j * rng.standard_normal(sh)) / math.sqrt(2.0)  # noqa: E731
    x = (o.freqs - F0) / F0
    xs = np.stack([x ** l for l in range(4)], 1)
    A0, D = cn(o.K, o.N, 4, 2, 2), 0.3 * cn(o.K, o.N, 4, 2, 2)
    al, be = rng.uniform(0, 1, (2, o.K, o.N, 4, 1, 1))

    def jones(iv):
        J = np.eye(2) + 0.1 * np.einsum("knlij,fl->fknij", A0 + D * np.sin(al * iv + 2 * math.pi * be), xs)
        return torch.from_numpy(J.astype(np.complex64)).to(dev)

    o.J = torch.stack([jones(iv) for iv in range(o.I)]).reshape(o.A, o.K, o.N, 2, 2)
    noise = torch.randn((o.A, o.K, o.N, 2, 2), generator=gen, device=dev, dtype=torch.complex64)
    o.J += 0.01 * noise
    o.J_prev = torch.stack([jones(iv - 1) for iv in range(o.I)]).reshape(o.A, o.K, o.N, 2, 2)
    o.flags = None
    if case["flagged"] > 0:
        o.flags = (rng.uniform(0, 1, (o.A, o.B)) < case["flagged"]).astype(np.uint8)
    if vis or coh:
        V = torch.empty(int(o.T.sum()) * o.B * 4, dtype=torch.complex64, device=dev) if vis else None
        C = torch.empty(int(o.T.sum()) * o.B * o.K, dtype=torch.complex64, device=dev) if coh else None
        v = k = 0
        for a, b, Ta in _groups(o):
            c = _coherencies(o, a, b, Ta, torch.complex64)
            n = (b - a) * o.B * Ta
            if coh:
                C[k:k + n * o.K] = c.reshape(-1)
                k += n * o.K
            if vis:
                m = torch.matmul(o.J[a:b][:, :, o.p], o.J[a:b][:, :, o.q].mH)  # [a, K, B, 2, 2]
                w = torch.einsum("abtk,akbij->abtij", c, m)
                w += 0.22 * w.abs().square().mean().sqrt() * torch.randn(w.shape, generator=gen, device=dev, dtype=torch.complex64)
                V[v:v + 4 * n] = w.reshape(-1)
                v += 4 * n
        o.V, o.C = V, C
    return o


def _real(x):
    return torch.view_as_real(x)


def _context(o, case, stream, **kw):
    T = o.T if len(set(o.T.tolist())) > 1 else int(o.T[0])
    return Calibrator(o.N, o.pq, o.K, o.freqs, o.basis, o.rho, n_intervals=o.I, samples=T, cuda_stream=stream.cuda_stream, **kw)


def _solver(case):
    return {"n_lm": case["n_lm"], "n_cg": case["n_cg"], "jupdate": JUPDATE[case["jupdate"]]}


def _rows(case, seed):
    """Training rows as the drivers make them: a drifting solution, its fit over frequency, the next solution."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    rand = lambda *sh: torch.randn(sh, generator=gen, device="cuda")  # noqa: E731
    eye = torch.tensor([1.0, 0, 0, 0, 0, 0, 1.0, 0], device="cuda")
    J = eye + 0.1 * rand(case["rows"], 8)
    X = torch.cat([J, J + 0.01 * rand(case["rows"], 8), torch.rand((case["rows"], 1), generator=gen, device="cuda")], 1)
    return X.contiguous(), (J + 0.02 * rand(case["rows"], 8)).contiguous()


def _weights(width, depth, seed):
    """A trained network's weights: the driver's initial ones with a last layer that is not zero any more."""
    w = init_weights(width, depth, seed)
    n = 8 * width + 8
    w[-n:-8] = 0.002 * np.random.default_rng(seed).standard_normal(8 * width).astype(np.float32)
    return w


def _point(o, seed):
    """Where L and its derivatives are taken: J off the truth, a direction, Y, Z, and the weights of a loss."""
    gen = torch.Generator(device="cuda").manual_seed(seed + 5)
    rand = lambda *sh, dt=torch.complex64: torch.randn(sh, generator=gen, device="cuda", dtype=dt)  # noqa: E731
    J = o.J + 0.05 * rand(*o.J.shape)
    eta = 0.1 * rand(*o.J.shape)
    Y = 0.1 * rand(*o.J.shape)
    Z = 0.1 * rand(o.I, o.K, o.M, o.N, 2, 2, dt=torch.complex128)
    return J, eta, Y, Z, torch.rand(o.A, generator=gen, device="cuda", dtype=torch.float64)


LR, DECAY, EARLIER = 1e-3, 1e-4, 3  # the driver's step; optimiser steps already taken


def prepare(case, seed):
    what = case["what"]
    if what == "train":
        net = WarmStartNet(case["width"], case["depth"], seed)
        st = {"what": what, "keep": net, "net": net.h, "stream": net.stream}
        capi.calib_mlp_set_weights(net.h, _weights(case["width"], case["depth"], seed))
        n = capi.calib_mlp_num_params(net.h)
        st["W"] = torch.empty(n, dtype=torch.float32, device="cuda")
        st["loss"] = torch.zeros(1, dtype=torch.float64, device="cuda")
        for k in range(EARLIER):
            X, T = _rows(case, seed * 100 + 1 + k)
            torch.cuda.synchronize()
            capi.calib_mlp_train_step(st["net"], X, T, LR, DECAY, st["loss"])
            torch.cuda.synchronize()
        st["X"], st["T"] = _rows(case, seed * 100)
        torch.cuda.synchronize()
        return st
    st = {"what": what, "stream": torch.cuda.Stream(), "iters": case.get("iters")}
    if what == "predict":
        o = _observation(case, seed, vis=False)
        st["cal"] = _context(o, case, st["stream"])
        st["out"] = torch.empty(int(o.T.sum()) * o.B * o.K, dtype=torch.complex64, device="cuda")
        st["o"] = o
        torch.cuda.synchronize()
        return st
    o = _observation(case, seed, vis=True, coh=what != "calibrate")
    st["o"] = o
    kw = _solver(case) if what in ("calibrate", "track") else {}
    cal = st["cal"] = _context(o, case, st["stream"], **kw)
    flags = None if o.flags is None else torch.from_numpy(o.flags).cuda()
    torch.cuda.synchronize()
    cal.set_data(_real(o.V), None if o.C is None else _real(o.C), flags)
    st["flags"] = flags
    st["J"] = torch.empty(cal.jones_shape, dtype=torch.complex64, device="cuda")
    if what in ("calibrate", "track"):
        st["Z"] = torch.empty(cal.z_shape, dtype=torch.complex128, device="cuda")
        o.C = None if what == "calibrate" else o.C
    if what == "track":
        Bt = torch.from_numpy(np.linalg.pinv(o.basis)).cuda().to(torch.complex128)  # the fit of the previous solution
        Jp = o.J_prev.reshape(o.I, o.P, o.K, o.N, 2, 2).to(torch.complex128)
        st["Z_prev"] = torch.einsum("mf,ifknab->ikmnab", Bt, Jp).contiguous()
        st["mlp"] = None
        if case["net"]:
            st["keep"] = WarmStartNet(256, 3, seed)
            st["mlp"] = st["keep"].h
            capi.calib_mlp_set_weights(st["mlp"], _weights(256, 3, seed))
    if what in ("gradient", "hessian", "loss"):
        st["at"], st["eta"], Y, Z, st["weight"] = _point(o, seed)
        st["L"] = torch.empty(o.A, dtype=torch.float64, device="cuda")
        if what != "hessian":  # the consensus state that the penalty holds J to
            torch.cuda.synchronize()
            cal.set_consensus(_real(Z), _real(Y))
            st["YZ"] = Y, Z
    if what == "loss":
        st["at"].requires_grad_(True)
    if what == "apply":
        st["out"] = torch.empty(o.V.numel(), dtype=torch.complex64, device="cuda")
    torch.cuda.synchronize()
    return st


def run(st):
    what = st["what"]
    with torch.cuda.stream(st["stream"]):
        if what == "train":
            capi.calib_mlp_train_step(st["net"], st["X"], st["T"], LR, DECAY, st["loss"])
            capi.calib_mlp_get_weights(st["net"], st["W"])
            return {"weights": st["W"], "loss": st["loss"].float()}
        o, ctx = st["o"], st["cal"].ctx
        if what == "calibrate":
            capi.calib_predict(ctx, o.uvw, o.sky, F0)
            capi.calib_reset(ctx)
            capi.calib_admm_iter(ctx, st["iters"], want_hist=False)
        if what == "track":
            capi.calib_set_data(ctx, _real(o.V), _real(o.C))
            capi.calib_warm_start(ctx, st["mlp"], _real(o.J_prev), _real(st["Z_prev"]))
            capi.calib_admm_iter(ctx, st["iters"], want_hist=False)
        if what in ("calibrate", "track"):
            capi.calib_get_solutions(ctx, _real(st["J"]), _real(st["Z"]))
            return {"J": st["J"], "Z": st["Z"].to(torch.complex64)}
        if what == "gradient":
            capi.calib_eval(ctx, _real(st["at"]), st["L"], None, _real(st["J"]))
            return {"L": st["L"].float(), "grad": st["J"]}
        if what == "loss":
            st["at"].grad = None
            L = admm_loss(st["at"], st["cal"])
            (L * st["weight"]).sum().backward()
            return {"L": L.detach().float(), "grad": st["at"].grad}
        if what == "hessian":
            capi.calib_hessvec(ctx, _real(st["at"]), _real(st["eta"]), _real(st["J"]))
            return st["J"]
        if what == "apply":
            capi.calib_set_data(ctx, _real(o.V), _real(o.C), st["flags"])
            capi.calib_set_initial(ctx, _real(o.J))
            capi.calib_residual(ctx, _real(st["out"]), None, 0)
            return st["out"]
        if what == "predict":
            capi.calib_predict(ctx, o.uvw, o.sky, F0)
            capi.calib_get_coherencies(ctx, _real(st["out"]))
            return st["out"]
    raise ValueError(what)


# ----------------------------------------------------------------------------- what a pass cannot do without

def _samples(case):
    """Unflagged visibilities of the batch (the mean over the draw of ragged samples and flags)."""
    mean_T = 0.5 * (case["Tmin"] + case["T"])
    return case["I"] * case["P"] * (case["N"] * (case["N"] - 1) / 2) * (1 - case["flagged"]) * mean_T


def work(case):
    what = case["what"]
    if what == "train":
        w, d, n = case["width"], case["depth"], case["rows"]
        params = 17 * w + (d - 1) * w * w + 8 * w + d * w + 8
        # forward and two products backward (none towards the inputs of the first layer); rows in, weights and both moments in and out
        return {"bytes": 4.0 * n * 25 + 28.0 * params, "flops": 6.0 * n * params - 2.0 * n * 17 * w}
    N, K, P, I, S, M = (float(case[k]) for k in ("N", "K", "P", "I", "S", "M"))
    A, B = I * P, N * (N - 1) / 2 * (1 - case["flagged"])
    vis, sol, z = _samples(case), 32 * A * K * N, 64 * I * K * M * N
    predict = vis * K * S * 8 + 30 * I * P * 0.5 * (case["Tmin"] + case["T"]) * N * K * S
    if what == "predict":
        return {"bytes": vis * 8 * K + 24 * I * case["T"] * N, "flops": predict}
    if what == "gradient" or what == "loss":
        return {"bytes": vis * (32 + 8 * K) + 4 * sol, "flops": vis * (64 * K + 8) + A * B * 184 * K}
    if what == "hessian":
        return {"bytes": vis * 8 * K + 3 * sol, "flops": min(vis * 64 * K, vis * 4 * K * K + A * B * 32 * K * K) + A * B * 248 * K}
    if what == "apply":
        return {"bytes": vis * (64 + 8 * K) + 2 * sol, "flops": vis * (32 * K + 120)}
    # sums over the samples of a baseline once, then per inner step a trial point's cost and gradient and the CG's Hessian products
    stats = vis * (32 * K + 4 * K * (K + 1))
    hess = min(248 * K + 32 * K * K, 64 * K * K - 32 * K)
    inner = A * B * (360 * K + 48 * K * K + case["n_cg"] * hess)
    once = predict + (vis * 60 * K if what == "track" else 0)
    data = vis * 32 + (vis * 8 * K if what == "track" else 0)
    return {"bytes": data + 2 * sol + z, "flops": once + stats + case["iters"] * case["n_lm"] * inner}


# ----------------------------------------------------------------------------- the same in 64 bits

def _agents(o, V=True):
    """(agent, V [B, T, 2, 2], C [B, T, K], J index pairs kept) of each agent in 64 bits, flagged baselines left out."""
    v = k = 0
    for a in range(o.A):
        n = o.B * int(o.T[a])
        keep = slice(None) if o.flags is None else torch.from_numpy(np.nonzero(o.flags[a] == 0)[0]).cuda()
        C = o.C[k:k + n * o.K].reshape(o.B, -1, o.K).to(torch.complex128)[keep]
        Va = o.V[v:v + 4 * n].reshape(o.B, -1, 2, 2).to(torch.complex128)[keep] if V else None
        yield a, Va, C, o.p[keep], o.q[keep]
        v, k = v + 4 * n, k + n * o.K


def _to_stations(C, X, J, p, q, K):
    """sum over baselines of conj(c) X J_q at station p and c X^H J_p at station q, [K, N, 2, 2]."""
    W = torch.einsum("btk,btij->kbij", C.conj(), X)
    out = torch.zeros_like(J)
    out.index_add_(1, p, W @ J[:, q])
    return out.index_add_(1, q, W.mH @ J[:, p])


def exact(case, seed):
    what = case["what"]
    if what in ("calibrate", "track"):
        return None  # hundreds of inner steps that each depend on the last
    if what == "train":
        return _exact_train(case, seed)
    if what == "predict":
        o = _observation(case, seed, vis=False)
        return torch.cat([_coherencies(o, a, b, Ta, torch.complex128).reshape(-1) for a, b, Ta in _groups(o)])
    o = _observation(case, seed, vis=True, coh=True)
    if what == "apply":
        out = []
        for a, V, C, p, q in _agents(o):
            J = o.J[a].to(torch.complex128)
            R = V - torch.einsum("btk,kbij->btij", C, J[:, p] @ J[:, q].mH)
            R = torch.linalg.inv(J[0, p])[:, None] @ R @ torch.linalg.inv(J[0, q]).mH[:, None]
            full = torch.zeros((o.B,) + R.shape[1:], dtype=R.dtype, device="cuda")
            full[slice(None) if o.flags is None else torch.from_numpy(np.nonzero(o.flags[a] == 0)[0]).cuda()] = R
            out.append(full.reshape(-1))
        return torch.cat(out)
    at, eta, Y, Z, weight = _point(o, seed)
    rho = torch.from_numpy(o.rho).cuda()[:, None, None, None]
    res, Ls = [], []
    for a, V, C, p, q in _agents(o):
        J, E = at[a].to(torch.complex128), eta[a].to(torch.complex128)
        if what == "hessian":
            dM = torch.einsum("btk,kbij->btij", C, E[:, p] @ J[:, q].mH + J[:, p] @ E[:, q].mH)
            res.append(_to_stations(C, dM, J, p, q, o.K) + 0.5 * rho * E)
            continue
        b = torch.from_numpy(o.basis[a % o.P]).cuda().to(torch.complex128)
        D, Ya = J - torch.einsum("m,kmnij->knij", b, Z[a // o.P]), Y[a].to(torch.complex128)
        R = V - torch.einsum("btk,kbij->btij", C, J[:, p] @ J[:, q].mH)
        Ls.append((R.abs() ** 2).sum() + (Ya.conj() * D).real.sum() + 0.5 * (rho * D.abs() ** 2).sum())
        res.append(-_to_stations(C, R, J, p, q, o.K) + 0.5 * Ya + 0.5 * rho * D)
    if what == "hessian":
        return torch.stack(res)
    L, grad = torch.stack(Ls), torch.stack(res)
    return {"L": L, "grad": 2.0 * weight[:, None, None, None, None] * grad if what == "loss" else grad}


def _exact_train(case, seed):
    w = torch.from_numpy(_weights(case["width"], case["depth"], seed)).cuda().double()
    m, v = torch.zeros_like(w), torch.zeros_like(w)
    dims = [17] + [case["width"]] * case["depth"] + [8]
    for t in range(1, EARLIER + 2):
        X, T = (x.double() for x in _rows(case, seed * 100 + (t if t <= EARLIER else 0)))
        wb = w.float().bfloat16().double().requires_grad_(True)  # the weights that the layers use
        h, at = X, 0
        for l, (i, n) in enumerate(zip(dims[:-1], dims[1:])):
            W, b = wb[at:at + i * n].reshape(n, i), wb[at + i * n:at + i * n + n]
            at += i * n + n
            h = h @ W.T + b
            h = torch.relu(h) if l < case["depth"] else h
        loss = ((X[:, :8] + h - T) ** 2).sum() / X.shape[0]
        (g,) = torch.autograd.grad(loss, wb)
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        w = w - LR * ((m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + 1e-8) + DECAY * w)
    return {"weights": w.detach(), "loss": loss.detach().reshape(1)}
