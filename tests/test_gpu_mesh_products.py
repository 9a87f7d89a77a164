"""The mesh products of float32 matrices (F P and P F^T + Q of eqns 7 and 11) summed in pairs of float32: the rounding
of the float64 sum wherever the pair holds enough of it, and the float64 sum itself elsewhere."""
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


def sparse(N, rng):
    """One to nine entries of both signs per row; row 3 empty."""
    rows = [np.sort(rng.choice(N, min(N, rng.integers(1, 10)), replace=False)) for _ in range(N)]
    rows[3] = rows[3][:0]
    rp = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int64)
    return rp, np.concatenate(rows).astype(np.int64), rng.standard_normal(rp[-1])


def check(right, rp, col, val, P, ld, q_kind=-1, Q=None):
    N = len(P)
    pad = np.zeros((N, ld), np.float32)
    pad[:, :N] = P
    t = lambda a: torch.from_numpy(a).cuda()
    out = torch.zeros(N, ld, dtype=torch.float32, device="cuda")
    B.kfx_spmm_packed(right, N, len(val), t(rp), t(col), t(val), t(pad), ld, out, ld, q_kind, None if Q is None else t(Q))
    got = out.cpu().numpy()[:, :N]
    M = (P.T if right else P).astype(np.float64)  # rows of M combined by F
    ref, mag = np.zeros((N, N)), np.zeros((N, N))
    with np.errstate(all="ignore"):
        for i in range(N):
            for k in range(rp[i], rp[i + 1]):
                ref[i] += val[k] * M[col[k]]
                mag[i] += np.abs(val[k] * M[col[k]])
        if right:
            ref, mag = ref.T.copy(), mag.T
        if q_kind >= 0:
            Qm = Q[0] * np.eye(N) if q_kind == 0 else np.diag(Q) if q_kind == 1 else Q
            ref, mag = ref + Qm, mag + np.abs(Qm)
        want = ref.astype(np.float32)
        fin = np.isfinite(want)
        assert np.array_equal(np.isnan(got), np.isnan(want))
        assert np.array_equal(got[~fin & ~np.isnan(want)], want[~fin & ~np.isnan(want)])
        # half a unit, ties to 2^-6 of one, and what the float64 reference itself has lost
        tol = (0.5 + 2.0 ** -6) * np.spacing(np.abs(want)) + 16 * 2.0 ** -53 * mag
        err = np.abs(got - ref)
        assert np.all(err[fin] <= tol[fin]), (err[fin] / tol[fin]).max()


@pytest.mark.parametrize("right", [0, 1])
@pytest.mark.parametrize("N,ld", [(5, 8), (50, 52), (50, 7000), (50, 14000), (2433, 2436)])
def test_float32_rounding_of_the_float64_sum(right, N, ld):
    rng = np.random.default_rng(N + ld)
    check(right, *sparse(N, rng), rng.standard_normal((N, N)).astype(np.float32), ld)


@pytest.mark.parametrize("right", [0, 1])
@pytest.mark.parametrize("e", [-147, -135, -126, -110, -95, 100, 118, 127])
def test_small_and_large_covariances(right, e):
    rng = np.random.default_rng(abs(e))
    N = 50
    rp, col, val = sparse(N, rng)
    P = np.ldexp(rng.uniform(-1, 1, (N, N)), e).astype(np.float32)
    check(right, rp, col, val, P, 52)
    if right:
        for kind, Q in ((0, np.full(1, 2.0 ** e)), (1, np.ldexp(rng.uniform(0, 1, N), e)),
                        (2, np.ldexp(rng.standard_normal((N, N)), e - 20))):
            check(right, rp, col, val, P, 52, kind, Q)


@pytest.mark.parametrize("right", [0, 1])
@pytest.mark.parametrize("bits", [12, 18, 24])
def test_sums_that_cancel(right, bits):
    """F takes differences of nearly equal rows: all but the last bits of the terms cancel."""
    rng = np.random.default_rng(bits)
    N = 48
    P = rng.standard_normal((N, N)).astype(np.float32)
    P[1::2] = (P[::2].astype(np.float64) * (1 + 2.0 ** -bits * rng.standard_normal((N // 2, N)))).astype(np.float32)
    rp = np.arange(0, 3 * N + 1, 3, dtype=np.int64)
    i = np.arange(N)
    col = np.stack([i // 2 * 2, i // 2 * 2 + 1, (i + 7) % N], 1).reshape(-1).astype(np.int64)
    a = rng.uniform(0.5, 1.5, N)
    val = np.stack([a, -a * (1 + 2.0 ** -bits * rng.standard_normal(N)), 2.0 ** -30 * rng.standard_normal(N)], 1).reshape(-1)
    check(right, rp, col, val, P.T.copy() if right else P, 52)


@pytest.mark.parametrize("right", [0, 1])
def test_entries_of_F_beyond_float32_and_values_that_are_not_finite(right):
    rng = np.random.default_rng(2)
    N = 40
    rp, col, val = sparse(N, rng)
    P = rng.standard_normal((N, N)).astype(np.float32)
    val[::7] *= 1e-42
    val[1::7] *= 1e-60
    check(right, rp, col, val, P, 40)
    big = (P * np.float32(1e-30)).astype(np.float32)
    val[::7] *= 1e82  # 1e40
    check(right, rp, col, val, big, 40)
    val[2::7] = 0.0
    P[5, 8], P[9, 1], P[20, 20] = np.inf, -np.inf, np.nan
    check(right, rp, col, val, P, 40)
