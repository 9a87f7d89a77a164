"""Performance cases of the filter, the smoother and the minimum-norm estimate.

A case is one call (or the filter + smoother pair) that a user of this package makes on a plan it
already holds, through solver.Plan, binding.kf_solve_host, binding.mne_solve or binding.mne_init.
The shapes are those of the package's own workloads (synth.py: the N = 384 float64 epoch, the
N = 5124 paper-scale mesh epoch, the N = 8196 benchmark, the batched epochs with N from 256 to
2048, the served requests with m = 306) with fewer time steps, since every step of an epoch costs
the same.  T, N and m of the drawn cases are spread over the same ranges, odd values included.

Inputs are synthetic, as synth.py draws them: a Gaussian lead field with depth-scaled columns, a few
active sources carrying 10-20 Hz sinusoids under a 0.4 Hz envelope, diagonal sensor noise; they are
drawn on the GPU from the seed.

The mixed path forms P_{t|T} in float32, so the float64 array of its diagonal holds float32 values;
such a program keeps it as float32 (the conversion is lossless).  Every other output stays as it is.
"""
from __future__ import annotations

import math
from functools import lru_cache

import numpy as np
import torch

from paper_1107_4192_gb300 import binding as B
from paper_1107_4192_gb300 import solver, synth

Q0 = 1e-2  # state-noise variance of every workload
SOLVES = {"mean": B.KF_SOLVE_FP64_MEAN, "tc": B.KF_SOLVE_FP64_TC, "fp64": B.KF_SOLVE_FP64}


def listed():
    return [
        # The smallest whole epoch: float64 throughout, the package's plain workload.  Launches and
        # dependent chains count.
        dict(name="epoch_fp64_N384", kind="epoch", prec="fp64", N=384, m=64, T=40, F="I", solve="fp64", ckpt=0),
        # A float64 mesh epoch large enough for the float64 units to count, ragged against 64.
        dict(name="epoch_fp64_N1026_mesh", kind="epoch", prec="fp64", N=1026, m=306, T=4, F="mesh", solve="fp64",
             ckpt=0),
        # Filtering alone (online estimates) of a small epoch of the batched workload.
        dict(name="filter_N640_m64_mesh", kind="filter", prec="mixed", N=640, m=64, T=40, F="mesh", solve="mean",
             ckpt=0),
        # Filtering alone at a middle size of the batched workload, random-walk dynamics.
        dict(name="filter_N1664_m128", kind="filter", prec="mixed", N=1664, m=128, T=24, F="I", solve="mean",
             ckpt=0),
        # The smallest served request, whole: filter and smoother with the server's default solve.
        dict(name="epoch_N1024_served", kind="epoch", prec="mixed", N=1024, m=306, T=20, F="mesh", solve="mean",
             ckpt=0),
        # A served request that enters and leaves through host memory.
        dict(name="host_N2048_served", kind="host", prec="mixed", N=2048, m=306, T=8, F="I", solve="mean", ckpt=0),
        # Smoothing alone with the float64-accurate gain at an odd size.
        dict(name="smooth_N1501_fp64tc", kind="smooth", prec="mixed", N=1501, m=128, T=8, F="I", solve="tc",
             ckpt=0),
        # The paper-scale mesh epoch, forward.
        dict(name="filter_N5124_mesh", kind="filter", prec="mixed", N=5124, m=306, T=6, F="mesh", solve="mean",
             ckpt=0),
        # The paper-scale mesh epoch, backward, in the server's checkpointed mode (covariances
        # between checkpoints are recomputed forward).
        dict(name="smooth_N5124_mesh_ckpt", kind="smooth", prec="mixed", N=5124, m=306, T=4, F="mesh", solve="mean",
             ckpt=2),
        # The benchmark workload, whole: N = 8196, random walk, float64-accurate smoother gain.
        dict(name="epoch_N8196_fp64tc", kind="epoch", prec="mixed", N=8196, m=306, T=4, F="I", solve="tc", ckpt=0),
        # Minimum-norm estimates of a recording (float64), the paper's comparison method.
        dict(name="mne_N5124_T200", kind="mne", N=5124, m=306, T=200),
        # The paper's initialisation: x0 and the dense state-noise covariance from the estimates.
        dict(name="mne_init_N8196_T300", kind="mne_init", N=8196, m=306, T=300),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["filter", "filter", "smooth", "smooth", "epoch", "host", "fp64", "mne", "mne_init"])
    m = rng.choice([64, 128, 306, rng.randint(33, 320)])
    if kind == "mne":
        return dict(kind="mne", N=_log_int(rng, 256, 8196), m=m, T=_log_int(rng, 20, 400))
    if kind == "mne_init":
        return dict(kind="mne_init", N=_log_int(rng, 256, 5200), m=m, T=_log_int(rng, 20, 300))
    F = rng.choice(["I", "mesh"])
    if kind == "fp64":
        N = _log_int(rng, 200, 1100)
        return dict(kind="epoch", prec="fp64", N=N, m=m, T=rng.randint(3, 12 if N < 600 else 4), F=F, solve="fp64",
                    ckpt=0)
    N = _log_int(rng, 256, 5200 if kind in ("filter", "smooth") else 2100)
    T = rng.randint(4, 32 if N < 1100 else 12 if N < 2200 else 5)
    ckpt = 2 if kind == "smooth" and rng.random() < 0.25 else 0
    return dict(kind=kind, prec="mixed", N=N, m=m, T=T, F=F, solve=rng.choice(["mean", "tc"]), ckpt=ckpt)


# ------------------------------------------------------------------------- inputs


@lru_cache(maxsize=8)
def _mesh(N):
    F = synth.mesh_coupling(synth.hemisphere_mesh(N))
    return F.rowptr, F.col, F.val


def _inputs(case, seed):
    """H, Y and R of one recording, on the GPU."""
    N, m, T = case["N"], case["m"], case["T"]
    g = torch.Generator(device="cuda").manual_seed(seed)
    rand = lambda *s: torch.rand(*s, generator=g, device="cuda", dtype=torch.float64)
    randn = lambda *s: torch.randn(*s, generator=g, device="cuda", dtype=torch.float64)
    H = randn(m, N) * torch.exp(-3.0 * rand(N))
    t = torch.arange(1, T + 1, device="cuda", dtype=torch.float64) / synth.SAMPLE_HZ
    envelope = torch.sin(2 * math.pi * 0.4 * t)
    Y = torch.zeros(T, m, device="cuda", dtype=torch.float64)
    for _ in range(3):
        active = torch.exp(-0.5 * (randn(N) * 6.0) ** 2) * rand(N)
        signal = torch.sin(2 * math.pi * (10.0 + 10.0 * rand(1)) * t) * envelope
        Y += signal[:, None] * (H @ active)[None, :]
    R = 0.5 + 1.5 * rand(m)
    Y += randn(T, m) * torch.sqrt(R)
    return H, Y, R


def _device_inputs(case, seed):
    N = case["N"]
    H, Y, R = _inputs(case, seed)
    dev = lambda a: torch.from_numpy(a).cuda()
    kind, F, rowptr, col, nnz = B.KF_F_IDENTITY, None, None, None, 0
    if case["F"] == "mesh":
        rp, c, v = _mesh(N)
        kind, F, rowptr, col, nnz = B.KF_F_CSR, dev(v), dev(rp), dev(c), int(rp[-1])
    return solver.DeviceInputs(kind, F, rowptr, col, nnz, B.KF_COV_SCALAR,
                               torch.tensor([Q0], dtype=torch.float64, device="cuda"), H, B.KF_COV_DIAG, R, Y,
                               torch.zeros(N, dtype=torch.float64, device="cuda"),
                               torch.eye(N, dtype=torch.float64, device="cuda"))


def prepare(case, seed):
    N, m, T, kind = case["N"], case["m"], case["T"], case["kind"]
    state = dict(case=case)
    if kind in ("mne", "mne_init"):
        state["H"], state["Y"], state["R"] = _inputs(case, seed)
        state["C"] = torch.ones(1, dtype=torch.float64, device="cuda")
        return state
    d = _device_inputs(case, seed)
    mixed = case["prec"] == "mixed"
    plan = solver.Plan.for_inputs(d, N, m, T, prec=B.KF_PREC_MIXED_BF16X3 if mixed else B.KF_PREC_FP64,
                                  solve_prec=SOLVES[case["solve"]], joseph_every=16 if mixed else 0,
                                  checkpoint_every=case["ckpt"])
    state["plan"] = plan
    if kind == "host":
        pin = lambda a: None if a is None else a.cpu().pin_memory()
        state["in"] = [pin(a) for a in (d.F, d.F_rowptr, d.F_col, d.Q, d.H, d.R, d.Y, d.x0, d.P0)]
        state["out"] = [torch.empty(T, N, dtype=torch.float64).pin_memory() for _ in range(4)]
        return state
    state["d"] = d
    if kind == "smooth":
        plan.filter(d)
    return state


# ------------------------------------------------------------------------- one pass


def run(state):
    case = state["case"]
    N, m, T, kind = case["N"], case["m"], case["T"], case["kind"]
    if kind == "mne":
        X = torch.empty(T, N, dtype=torch.float64, device="cuda")
        B.mne_solve(state["H"], state["C"], B.KF_COV_SCALAR, state["R"], B.KF_COV_DIAG, state["Y"], N, m, T, 1.0, X)
        return {"X": X}
    if kind == "mne_init":
        x0 = torch.empty(N, dtype=torch.float64, device="cuda")
        Q = torch.empty(N, N, dtype=torch.float64, device="cuda")
        B.mne_init(state["H"], state["C"], B.KF_COV_SCALAR, state["R"], B.KF_COV_DIAG, state["Y"], N, m, T, 1.0, None,
                   x0, Q)
        return {"x0": x0, "Q": Q}
    smoothed_diag = (lambda v: v.float()) if case["prec"] == "mixed" else (lambda v: v)
    plan = state["plan"]
    if kind == "host":
        xf, pf, xs, ps = state["out"]
        B.kf_solve_host(plan.handle, *state["in"], xf, pf, xs, ps)
        return {"x_filt": xf, "diagP_filt": pf, "x_smooth": xs, "diagP_smooth": smoothed_diag(ps)}
    out = {}
    if kind in ("filter", "epoch"):
        out["x_filt"], out["diagP_filt"] = plan.filter(state["d"])
    if kind in ("smooth", "epoch"):
        x, p, _ = plan.smooth()
        out["x_smooth"], out["diagP_smooth"] = x, smoothed_diag(p)
    return out


# ------------------------------------------------------------------------- what a pass needs


def work(case):
    N, m, T, kind = case["N"], case["m"], case["T"], case["kind"]
    if kind in ("mne", "mne_init"):
        # lambda H H^T (lower triangle), its Cholesky, two triangular solves with T right-hand sides, W H
        flops = m * m * N + m ** 3 / 3 + 2 * m * m * T + 2 * m * N * T
        nbytes = 8 * (m * N + T * m + T * N)
        if kind == "mne_init":
            flops += N * N * (T - 1)
            nbytes = 8 * (m * N + T * m + N + N * N)
        return {"bytes": nbytes, "flops": flops}
    nnz = 7 if case["F"] == "mesh" else 0
    word = 4 if case["prec"] == "mixed" else 8
    # filter step: P H^T, the lower triangles of H P H^T and of the update, Cholesky of S, one triangular
    # solve; F P F^T.  Smoother step: inverse of P_{t+1|t} (N^3), J D and the lower triangle of (J D) J^T.
    filt = 2 * m * N * N + m * m * N + m ** 3 / 3 + m * m * N + m * N * N + 4 * nnz * N * N
    smooth = 4 * N ** 3 + 4 * N * N + 2 * nnz * N * N
    means = 8 * 2 * T * N  # a mean and a variance per source and step
    store = word * T * N * N  # P_{t|t}: the filter's result for the smoother
    if kind == "filter":
        return {"bytes": 8 * (N * N + m * N + T * m) + store + means, "flops": T * filt}
    if kind == "smooth":
        return {"bytes": store + means, "flops": (T - 1) * smooth}
    return {"bytes": 8 * (N * N + m * N + T * m) + 2 * means, "flops": T * filt + (T - 1) * smooth}


# ------------------------------------------------------------------------- 64-bit reference


def _exact_mne(case, seed):
    H, Y, R = _inputs(case, seed)
    G = H @ H.T + torch.diag(R)
    return torch.cholesky_solve(Y.T, torch.linalg.cholesky(G)).T @ H


def exact(case, seed):
    N, T, kind = case["N"], case["T"], case["kind"]
    if kind == "mne":
        return {"X": _exact_mne(case, seed)}
    if kind == "mne_init":
        X = _exact_mne(case, seed)
        D = X[1:] - X[:-1]
        D = D - D.mean(0)
        return {"x0": X[0].clone(), "Q": D.T @ D / (T - 2)}
    H, Y, R = _inputs(case, seed)
    F = None
    if case["F"] == "mesh":
        rp, c, v = (torch.from_numpy(np.asarray(a)).cuda() for a in _mesh(N))
        F = torch.sparse_csr_tensor(rp, c, v, size=(N, N), dtype=torch.float64)
    left = (lambda A: A) if F is None else (lambda A: F @ A)  # F A
    right = (lambda A: A) if F is None else (lambda A: (F @ A.T).T)  # A F^T

    def predict(P):
        Pn = right(left(P)).clone()
        Pn.diagonal().add_(Q0)
        return Pn

    x = torch.zeros(N, dtype=torch.float64, device="cuda")
    P = torch.eye(N, dtype=torch.float64, device="cuda")
    xp, xf, Pf = [], [], []
    for t in range(T):
        x = left(x[:, None])[:, 0]
        P = predict(P)
        xp.append(x)
        U = P @ H.T
        L = torch.linalg.cholesky(H @ U + torch.diag(R))
        Z = torch.linalg.solve_triangular(L, U.T, upper=False)
        nu = torch.linalg.solve_triangular(L, (Y[t] - H @ x)[:, None], upper=False)
        x = x + (Z.T @ nu)[:, 0]
        P = P - Z.T @ Z
        xf.append(x)
        Pf.append(P)
    filt = {"x_filt": torch.stack(xf), "diagP_filt": torch.stack([p.diagonal().clone() for p in Pf])}
    if kind == "filter":
        return filt
    xs, Ps = [xf[-1]], [Pf[-1].diagonal().clone()]
    S = Pf[-1]
    for t in range(T - 2, -1, -1):
        Pn = predict(Pf[t])
        J = torch.cholesky_solve(left(Pf[t]), torch.linalg.cholesky(Pn)).T
        xs.append(xf[t] + J @ (xs[-1] - xp[t + 1]))
        S = Pf[t] + J @ (S - Pn) @ J.T
        Ps.append(S.diagonal().clone())
    smooth = {"x_smooth": torch.stack(xs[::-1]), "diagP_smooth": torch.stack(Ps[::-1])}
    return smooth if kind == "smooth" else {**filt, **smooth}
