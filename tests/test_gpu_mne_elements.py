"""Minimum-norm estimates element by element (eqn 5): every source and sample keeps float64 accuracy of its own, however
large the others are."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1107_4192_gb300 import binding as B  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1107_4192_gb300 import build
    build.build()
    B.lib()


def solve(H, R, Y, lam=1.3, c=None):
    m, N = H.shape
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    X = torch.empty(len(Y), N, dtype=torch.float64, device="cuda")
    B.mne_solve(t(H), t(np.ones(1) if c is None else c), 0 if c is None else 1, t(R), 1, t(Y), N, m, len(Y), lam, X)
    return X.cpu().numpy()


def reference(H, R, Y, lam=1.3):
    G = lam * H @ H.T + np.diag(R)
    V = np.linalg.solve(G, Y.T)
    V += np.linalg.solve(G, Y.T - G @ V)
    return lam * V.T @ H


@pytest.mark.parametrize("small", [1e-8, 1e-20, 1e-40])
@pytest.mark.parametrize("N,m,T", [(60, 16, 4), (700, 97, 33), (300, 306, 5)])
def test_groups_of_sensors_of_unequal_signal(N, m, T, small):
    """Two groups of sensors, each with sources of its own; the second group's samples are smaller by up to 1e40.  The
    groups do not mix, so each is the estimate from its own sensors alone.  Per source over the samples, 1e-11 for
    the conditioning of G; per element 1e-9, an element being able to cancel by a factor 100 against its terms."""
    rng = np.random.default_rng(N)
    H, R, Y = rng.standard_normal((m, N)), rng.uniform(0.5, 2, m), rng.standard_normal((T, m))
    a, n = m // 2, N // 3
    H[:a, n:] = 0.0
    H[a:, :n] = 0.0
    Y[:, a:] *= small
    X = solve(H, R, Y)
    ref = np.concatenate([reference(H[:a, :n], R[:a], Y[:, :a]), reference(H[a:, n:], R[a:], Y[:, a:])], 1)
    assert (np.linalg.norm(X - ref, axis=0) / np.linalg.norm(ref, axis=0)).max() <= 1e-11
    terms = np.abs(ref) + 0.01 * np.sqrt((ref ** 2).mean(0))
    assert (np.abs(X - ref) / terms).max() <= 1e-9


@pytest.mark.parametrize("noise", [1e8, 1e16, 1e30])
def test_sources_that_only_weakly_weighted_sensors_see(noise):
    """Bad channels, given a large noise variance, are the only ones to see some of the sources."""
    rng = np.random.default_rng(1)
    N, m, T, bad, n = 200, 40, 6, 5, 30
    H, R, Y = rng.standard_normal((m, N)), rng.uniform(0.5, 2, m), rng.standard_normal((T, m))
    H[:-bad, -n:] = 0.0
    H[-bad:, :-n] = 0.0
    R[-bad:] = noise
    X = solve(H, R, Y)
    ref = np.concatenate([reference(H[:-bad, :-n], R[:-bad], Y[:, :-bad]), reference(H[-bad:, -n:], R[-bad:], Y[:, -bad:])], 1)
    assert (np.linalg.norm(X - ref, axis=0) / np.linalg.norm(ref, axis=0)).max() <= 1e-11


def test_zero_samples_and_zero_sources():
    rng = np.random.default_rng(3)
    H, R, Y = rng.standard_normal((33, 70)), rng.uniform(0.5, 2, 33), rng.standard_normal((9, 33))
    H[:, 40:50] = 0.0
    Y[4] = 0.0
    X, ref = solve(H, R, Y), reference(H, R, Y)
    assert np.all(X[4] == 0.0) and np.all(X[:, 40:50] == 0.0)
    assert np.abs(X - ref).max() <= 1e-11 * np.abs(ref).max()


def test_a_sample_that_is_not_finite_stays_in_its_row():
    rng = np.random.default_rng(4)
    H, R, Y = rng.standard_normal((40, 300)), rng.uniform(0.5, 2, 40), rng.standard_normal((7, 40))
    good = solve(H, R, Y)
    Y[2, 11], Y[5, 0] = np.nan, np.inf
    X = solve(H, R, Y)
    bad = np.isin(np.arange(7), [2, 5])
    assert not np.isfinite(X[bad]).any()
    assert np.array_equal(X[~bad], good[~bad])
