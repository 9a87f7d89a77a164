"""The one-launch factorisation of the innovation covariance (eqn 8) at the edges of its tiles, through
the C ABI against the float64 oracle, and its failure reports.

Sizes: one row, a tile less / more one, several tiles with ragged ends, and both sides of the largest m it
takes (above it block kernels do the same).  Tolerance: the float64 path's 1e-10 on means and diag P.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1107_4192_gb300 import binding as B  # noqa: E402
from paper_1107_4192_gb300 import solver, synth  # noqa: E402
from tests.helpers import diag_of, rel_err_elementwise, rel_err_per_step, run_oracle  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1107_4192_gb300 import build
    build.build()
    B.lib()


@pytest.mark.parametrize("N,m", [(40, 1), (40, 31), (40, 32), (40, 33), (60, 64), (60, 65), (130, 97), (90, 306),
                                 (64, 960), (64, 961)])
def test_filter_at_tile_edges(N, m):
    prob = synth.random_walk_problem(N, m, 3, seed=N + m)
    out, ref = solver.run(prob, prec=B.KF_PREC_FP64), run_oracle(prob)
    assert rel_err_per_step(out["x_filt"], ref["x_filt"]) <= 1e-10
    assert rel_err_elementwise(out["diagP_filt"], diag_of(ref["P_filt"])) <= 1e-10


def _filter(plan, d, T, N):
    x = torch.empty(T, N, dtype=torch.float64, device="cuda")
    return B.kf_filter(plan.handle, d.F, d.F_rowptr, d.F_col, d.Q, d.H, d.R, d.Y, d.x0, d.P0, x, raise_on_error=False) + (x,)


@pytest.mark.parametrize("prec,solve", [(B.KF_PREC_FP64, B.KF_SOLVE_FP64), (B.KF_PREC_MIXED_BF16X3, B.KF_SOLVE_FP32)])
def test_failure_in_a_later_tile_then_recovery(prec, solve):
    """A singular S whose bad pivot lies in the third tile, then a non-finite sample, then good data on
    the same plan: the reports are those of the block algorithm, and nothing is left behind."""
    N, m, T = 150, 100, 3
    prob = synth.random_walk_problem(N, m, T, seed=9)
    good = solver.upload(prob)
    with solver.Plan.for_inputs(good, N, m, T, prec=prec, solve_prec=solve) as plan:
        st, step, x0 = _filter(plan, good, T, N)
        assert st == B.KF_OK
        bad = solver.upload(prob)
        bad.H[80:] = 0.0
        bad.R = torch.zeros_like(bad.R)
        st, step, _ = _filter(plan, bad, T, N)
        assert st == B.KF_ERR_NOT_PD and step == 1
        nan = solver.upload(prob)
        nan.Y[1, 70] = float("nan")
        st, step, _ = _filter(plan, nan, T, N)
        assert st == B.KF_ERR_NUMERIC and step == 2
        st, step, x1 = _filter(plan, good, T, N)
        assert st == B.KF_OK and torch.equal(x0, x1)


@pytest.mark.parametrize("N,m,T,mesh", [(33, 5, 3, True), (320, 40, 3, False), (1536, 20, 2, False), (1537, 20, 2, False)])
def test_float64_gain_on_both_sides_of_the_direct_size(N, m, T, mesh):
    """Float64 smoother with the one-launch factor and inverse of P_{t+1|t} and, above 1536 sources, with the
    block kernels; Joseph form every second step."""
    prob = synth.mesh_problem(N, m, T, seed=N, identity_F=not mesh)
    out, ref = solver.run(prob, prec=B.KF_PREC_FP64, joseph_every=2), run_oracle(prob)
    for k, tol in (("x_filt", 1e-10), ("x_smooth", 1e-10)):
        assert rel_err_per_step(out[k], ref[k]) <= tol
    for k, r in (("diagP_filt", "P_filt"), ("diagP_smooth", "P_smooth")):
        assert rel_err_elementwise(out[k], diag_of(ref[r])) <= 1e-10


def test_float64_gain_reports_a_singular_prediction():
    """P_{t+1|t} singular (Q = 0, P0 of low rank): the smoother's factor reports the step, and the plan works again."""
    N, m, T = 100, 8, 3
    prob = synth.random_walk_problem(N, m, T, seed=3)
    good = solver.upload(prob)
    with solver.Plan.for_inputs(good, N, m, T) as plan:
        st, _, _ = _filter(plan, good, T, N)
        x0 = plan.smooth()[0]
        bad = solver.upload(prob)
        bad.Q = torch.zeros_like(bad.Q)
        bad.P0 = torch.diag(torch.cat([torch.ones(70), torch.full((N - 70,), 1e-300)]).double()).cuda()
        bad.P0[80:, :] = 0
        st, step, x = _filter(plan, bad, T, N)
        if st == B.KF_OK:
            st, step = B.fis_smooth(plan.handle, x, raise_on_error=False)
        assert st in (B.KF_ERR_NOT_PD, B.KF_ERR_NUMERIC)
        st, _, _ = _filter(plan, good, T, N)
        assert st == B.KF_OK and torch.equal(plan.smooth()[0], x0)


@pytest.mark.parametrize("N,m,T,sensors,sources", [(300, 20, 5, 0, 0), (700, 64, 40, 6, 0), (130, 129, 3, 0, 8),
                                                   (900, 120, 60, 4, 4), (40, 1537, 3, 0, 0)])
def test_mne_with_sensors_and_sources_in_different_units(N, m, T, sensors, sources):
    """The minimum-norm products on slices keep float64 accuracy when sensors (rows) or sources (columns) are
    scaled apart by up to e^12 and e^16; per-source error, 1e-11 for the conditioning of G."""
    rng = np.random.default_rng(N + m)
    u, c = np.exp(rng.uniform(-sensors, sensors, m)), np.exp(rng.uniform(-sources, sources, N))
    H = rng.standard_normal((m, N)) * u[:, None] / np.sqrt(c)
    R, Y = rng.uniform(0.5, 2, m) * u ** 2, rng.standard_normal((T, m)) * u
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    X = torch.empty(T, N, dtype=torch.float64, device="cuda")
    B.mne_solve(t(H), t(c), 1, t(R), 1, t(Y), N, m, T, 1.3, X)
    # the reference in extended precision: float64 solves of the balanced system, refined (with m much larger than
    # N a float64 solve alone is off by the tolerance)
    Hl = H.astype(np.longdouble) / u[:, None]
    G = 1.3 * (Hl * c) @ Hl.T + np.diag(R / u ** 2).astype(np.longdouble)
    rhs, V = (Y / u).T.astype(np.longdouble), np.zeros((m, T), np.longdouble)
    for _ in range(4):
        V = V + np.linalg.solve(G.astype(np.float64), (rhs - G @ V).astype(np.float64))
    ref = (1.3 * V.T @ (Hl * c)).astype(np.float64)
    err = np.linalg.norm(X.cpu().numpy() - ref, axis=0) / np.linalg.norm(ref, axis=0)
    assert err.max() <= 1e-11
