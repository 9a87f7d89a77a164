"""The one-launch factorisation of the innovation covariance (eqn 8) bit for bit against the block kernels it stands
for and against correctly rounded square roots and reciprocals, and the filter and smoother around its largest size.
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


def factor(blocks, S, nu):
    m = len(S)
    dS, dL = torch.from_numpy(S.copy()).cuda(), torch.full((m, m), float("nan"), dtype=torch.float64, device="cuda")
    dn = torch.from_numpy(nu.copy()).cuda()
    st, fi = B.kfx_innovation_factor(blocks, m, dS, m, dL, dn)
    return st, fi, np.tril(dS.cpu().numpy()), dL.cpu().numpy(), dn.cpu().numpy()


@pytest.mark.parametrize("m", [1, 31, 32, 33, 64, 97, 306, 961, 1535, 1536])
@pytest.mark.parametrize("spread", [0.0, 12.0])
def test_same_bits_as_the_block_kernels(m, spread):
    rng = np.random.default_rng(m)
    G = rng.standard_normal((m, m + 5)) * np.exp(rng.uniform(-spread, spread, (m, 1)))
    S = G @ G.T + np.diag(rng.uniform(0.5, 2.0, m))
    S = 0.5 * (S + S.T)
    nu = rng.standard_normal(m)
    one, blk = factor(0, S, nu), factor(1, S, nu)
    assert one[:2] == (0, -1) and blk[:2] == (0, -1)
    for a, b in zip(one[2:], blk[2:]):
        assert np.array_equal(a, b)


def test_pivots_are_correctly_rounded():
    """L_ii = sqrt(S_ii) and its reciprocal, both rounded to nearest: random mantissas, those next to powers of four
    and of all-ones roots, inside and outside the range of the short form (2^-100 to 2^100)."""
    m = 1536
    rng = np.random.default_rng(0)
    d = rng.uniform(0.5, 2.0, m) * 2.0 ** rng.integers(-99, 100, m)
    k = np.arange(-45, 45)
    d[0:90] = np.nextafter(4.0 ** k, 0)
    d[90:180] = np.nextafter(4.0 ** k, 9e99)
    d[180:270] = 2.0 * 4.0 ** k
    root = np.nextafter(2.0, 0) * 2.0 ** k[10:80]
    d[270:340] = root * root
    d[340:410] = np.nextafter(root * root, 9e99)
    d[410:480] = np.nextafter(root * root, 0)
    d[480:700] = rng.uniform(0.5, 2.0, 220) * 2.0 ** np.concatenate([rng.integers(-1000, -100, 110), rng.integers(100, 1000, 110)])
    d[700:704] = [5e-324, 2.0 ** -1022, 1.7e308, 1.0]
    st, fi, L, X, nu = factor(0, np.diag(d), np.ones(m))
    assert (st, fi) == (0, -1)
    r = np.sqrt(d)
    assert np.array_equal(np.diag(L), r)
    assert np.array_equal(np.diag(X), 1.0 / r)
    assert np.array_equal(nu, 1.0 / r)


@pytest.mark.parametrize("bad", [0, 31, 32, 100, 305])
def test_first_bad_pivot_is_reported(bad):
    S = np.eye(306)
    S[bad, bad] = -1.0
    S[305, 305] = 0.0
    for blocks in (0, 1):
        assert factor(blocks, S, np.ones(306))[:2] == (B.KF_ERR_NOT_PD, bad)


@pytest.mark.parametrize("m", [1536, 1537])
@pytest.mark.parametrize("prec,solve,tol_x,tol_d", [(B.KF_PREC_FP64, B.KF_SOLVE_FP64, 1e-10, 1e-10),
                                                    (B.KF_PREC_MIXED_BF16X3, B.KF_SOLVE_FP64_MEAN, 1e-4, 1e-3)])
def test_filter_on_both_sides_of_the_largest_m(m, prec, solve, tol_x, tol_d):
    """m = 1536 in one launch, 1537 with the block kernels; Joseph form every second step.  The paths' tolerances."""
    prob = synth.random_walk_problem(64, m, 3, seed=m)
    out, ref = solver.run(prob, prec=prec, solve_prec=solve, joseph_every=2), run_oracle(prob)
    assert rel_err_per_step(out["x_filt"], ref["x_filt"]) <= tol_x
    assert rel_err_elementwise(out["diagP_filt"], diag_of(ref["P_filt"])) <= tol_d
    assert rel_err_per_step(out["x_smooth"], ref["x_smooth"]) <= tol_x


@pytest.mark.parametrize("prec,solve", [(B.KF_PREC_FP64, B.KF_SOLVE_FP64), (B.KF_PREC_MIXED_BF16X3, B.KF_SOLVE_FP64_TC)])
def test_smoother_reports_an_indefinite_prediction(prec, solve):
    """P0 indefinite on two sources that no sensor sees, Q = 0: the filter's diagonals stay positive, the smoother's
    factor of P_{3|2} meets the pivot 1 - 2 * 2 and reports step 3; the plan then works on good data."""
    N, m, T = 100, 8, 3
    prob = synth.random_walk_problem(N, m, T, seed=3)
    good, bad = solver.upload(prob), solver.upload(prob)
    bad.H[:, 70:72] = 0.0
    bad.Q = torch.zeros_like(bad.Q)
    bad.P0 = torch.eye(N, dtype=torch.float64, device="cuda")
    bad.P0[70, 71] = bad.P0[71, 70] = 2.0
    with solver.Plan.for_inputs(good, N, m, T, prec=prec, solve_prec=solve) as plan:
        plan.filter(good)
        x0 = plan.smooth()[0]
        plan.filter(bad)
        st, step = B.fis_smooth(plan.handle, torch.empty_like(x0), raise_on_error=False)
        assert (st, step) == (B.KF_ERR_NOT_PD, 3)
        plan.filter(good)
        assert torch.equal(plan.smooth()[0], x0)
