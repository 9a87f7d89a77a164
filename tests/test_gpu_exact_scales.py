"""The float64-accurate inverse (eqn 11) of matrices whose rows differ in scale: sources with unequal variances, as a
diagonal Q or P0 (depth weighting, mixed units) makes them."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1107_4192_gb300 import binding as B  # noqa: E402
from paper_1107_4192_gb300 import solver, synth  # noqa: E402
from tests.helpers import rel_err_per_step  # noqa: E402
from tests.test_gpu_exact import spd32  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1107_4192_gb300 import build
    build.build()
    B.lib()


def inverse(A):
    n = len(A)
    X = torch.zeros(n, n, dtype=torch.float64, device="cuda")
    assert B.kfx_spd_inverse(2, n, torch.from_numpy(A).cuda(), n, X, n) == (0, -1)
    return X.cpu().numpy()


def accurate_inverse(A):
    """Balanced float64 inverse: about 1e-14 relative to sqrt(X_ii X_jj) for a balanced condition number of 100."""
    d = 1.0 / np.sqrt(np.diag(A).astype(np.float64))
    return np.linalg.inv(A.astype(np.float64) * d[:, None] * d) * d[:, None] * d


@pytest.mark.parametrize("n", [5, 129, 300])
def test_powers_of_two_leave_the_digits_alone(n):
    """A scaled by powers of two on both sides gives the inverse scaled by them, bit for bit."""
    A = spd32(n, 100.0, n)
    e = np.random.default_rng(n).integers(-16, 17, n)
    D = np.ldexp(np.float32(1.0), e).astype(np.float32)
    X, Xs = inverse(A), inverse(A * D[:, None] * D)
    D = D.astype(np.float64)
    assert np.array_equal(Xs * D[:, None] * D, X)


@pytest.mark.parametrize("n,spread", [(300, 1e3), (300, 1e6), (700, 1e10), (1601, 1e6)])
def test_refined_inverse_with_rows_of_unequal_scale(n, spread):
    """P = A + diag(q) with q spread over many orders of magnitude: every element to float64 accuracy relative to
    sqrt(X_ii X_jj).  The balanced matrix has a condition number of about 100, so the bound is that of equal scales."""
    rng = np.random.default_rng(n)
    A = spd32(n, 100.0, n).astype(np.float64)
    q = np.exp(rng.uniform(0.0, np.log(spread), n))
    P = (A * np.sqrt(q)[:, None] * np.sqrt(q)).astype(np.float32)
    P = np.tril(P) + np.tril(P, -1).T
    X, ref = inverse(P), accurate_inverse(P)
    s = np.sqrt(np.diag(ref))
    assert np.abs((X - ref) / s[:, None] / s).max() <= 1e-12


def test_refined_inverse_of_a_matrix_with_a_large_diagonal():
    """A small dense part and a diagonal spread over 1e8: small rows next to large ones."""
    n = 300
    rng = np.random.default_rng(7)
    A = spd32(n, 100.0, 3).astype(np.float64) + np.diag(np.exp(rng.uniform(0.0, np.log(1e8), n)))
    P = A.astype(np.float32)
    P = np.tril(P) + np.tril(P, -1).T
    X, ref = inverse(P), accurate_inverse(P)
    s = np.sqrt(np.diag(ref))
    assert np.abs((X - ref) / s[:, None] / s).max() <= 1e-12


def test_smoother_with_a_diagonal_Q_over_eight_orders():
    """Smoothed means with Q and P0 diagonal and spread over 1e8, against the same filter with the float64 CUDA-core
    solve; each source in units of its prior deviation, 1e-10 as for the solves' agreement with equal variances."""
    N, m, T = 300, 40, 4
    prob = synth.mesh_problem(N, m, T, seed=5, identity_F=True)
    w = np.exp(np.random.default_rng(1).uniform(np.log(1e-4), np.log(1e4), N))
    d = solver.upload(prob)
    d.q_kind, d.Q = B.KF_COV_DIAG, torch.from_numpy(1e-2 * w).cuda()
    d.P0 = torch.diag(torch.from_numpy(w)).cuda()
    d.H = d.H / torch.from_numpy(np.sqrt(w)).cuda()
    xs = []
    for solve in (B.KF_SOLVE_FP64, B.KF_SOLVE_FP64_TC):
        with solver.Plan.for_inputs(d, N, m, T, prec=B.KF_PREC_MIXED_BF16X3, solve_prec=solve) as plan:
            plan.filter(d)
            xs.append(plan.smooth()[0].cpu().numpy() / np.sqrt(w))
    assert rel_err_per_step(xs[1], xs[0]) <= 1e-10
