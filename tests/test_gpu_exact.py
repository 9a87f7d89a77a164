"""The exact-slice tensor-core product and the float64-accurate inverse built on it, through the
C ABI (include/kfmeg_kernels.h).

 - kfx_gemm_exact against an independent numpy restatement of the slicing scheme (integer slices
   below each row's largest magnitude, exact integer level sums, one rounding at the end): the
   GPU must reproduce it to a few units in the last place, which pins the slicing, the exact
   accumulation and the scaling;
 - the same product against the true product of the float64 inputs (computed in extended
   precision) within the scheme's error bound;
 - kfx_spd_inverse (float32-class factor refined to float64 accuracy) against the float64
   CUDA-core solve (kfx_posv_right, itself checked against numpy) at N in {257, 1024, 2048}:
   the smoother-gain inverse of eqn 11 at float64 accuracy.
"""
import math

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


def rne_shift(a, s):
    """a / 2^s rounded to nearest, ties to even, for int64 arrays."""
    return (a + (1 << (s - 1)) - 1 + ((a >> s) & 1)) >> s


def slices_ref(X, S):
    """Row exponents e (max |X[r]| < 2^e) and integer slices q_p with
    X[r] ~= 2^(e_r - 7) sum_p 2^(-8p) q_p[r]: the signed base-256 digits (rounded to nearest,
    ties to even) of X rounded to the grid 2^(e_r - 7 - 8(S - 1))."""
    X = np.asarray(X, np.float64)
    mx = np.abs(X).max(axis=1)
    e = np.where(mx > 0, np.frexp(mx)[1], 0).astype(np.int64)
    Xi = np.rint(np.ldexp(X, (7 + 8 * (S - 1) - e)[:, None])).astype(np.int64)
    qs = []
    for p in range(S):
        sp = 8 * (S - 1 - p)
        q = rne_shift(Xi, sp) if sp > 0 else Xi.copy()
        assert np.abs(q).max(initial=0) <= 128
        Xi = Xi - (q << sp)
        qs.append(q)
    return e, qs


def exact_sliced_product(A, Bm, L):
    """Correctly rounded value of the sliced product keeping slice levels < L."""
    ea, qa = slices_ref(A, L)
    eb, qb = slices_ref(Bm, L)
    M, N = A.shape[0], Bm.shape[0]
    total = np.zeros((M, N), dtype=object)
    for lvl in range(L):
        V = sum(qa[a] @ qb[lvl - a].T for a in range(lvl + 1))  # exact int64
        total = total + V.astype(object) * (1 << (8 * (L - 1 - lvl)))
    out = np.empty((M, N))
    for i in range(M):
        for j in range(N):
            out[i, j] = math.ldexp(float(total[i, j]), int(ea[i] + eb[j]) - 14 - 8 * (L - 1))
    return out, ea, eb


@pytest.mark.parametrize("levels", [4, 5, 6, 7])
@pytest.mark.parametrize("M,N,K", [(130, 70, 300), (256, 192, 1024), (1, 1, 1), (129, 65, 33), (70, 130, 3000)])
def test_exact_product_matches_the_scheme(levels, M, N, K):
    rng = np.random.default_rng(M + N + K + levels)
    A = rng.standard_normal((M, K)) * np.exp(rng.uniform(-4, 4, (M, 1))) * np.exp(rng.uniform(-3, 3, (M, K)))
    Bm = rng.standard_normal((N, K)) * np.exp(rng.uniform(-4, 4, (N, 1)))
    ref, ea, eb = exact_sliced_product(A, Bm, levels)
    C = torch.zeros(M, N, dtype=torch.float64, device="cuda")
    B.kfx_gemm_exact(levels, M, N, K, 1.0, torch.from_numpy(A).cuda(), K, torch.from_numpy(Bm).cuda(), K, 0.0, 0.0,
                     C, N)
    got = C.cpu().numpy()
    # two roundings (the 64-bit level sums to float64) against one: a few ulp of the tile scale
    scale = np.ldexp(1.0, (ea[:, None] + eb[None, :]).astype(np.int64))
    assert np.all(np.abs(got - ref) <= 2.0 ** -50 * scale * max(1, K) ** 0.0 + 4 * np.spacing(np.abs(ref)))


@pytest.mark.parametrize("levels", [4, 5, 6, 7])
def test_exact_product_accuracy_and_epilogue(levels):
    """Against the true product (extended precision); alpha, beta and the delta on the diagonal."""
    rng = np.random.default_rng(7 + levels)
    M, N, K = 200, 200, 700
    A = rng.standard_normal((M, K))
    Bm = rng.standard_normal((N, K))
    C0 = rng.standard_normal((M, N))
    true = (A.astype(np.longdouble) @ Bm.astype(np.longdouble).T).astype(np.longdouble)
    ref = (-0.5 * true + 2.0 * C0.astype(np.longdouble) + np.eye(M, dtype=np.longdouble) * 3.0).astype(np.float64)
    C = torch.from_numpy(C0.copy()).cuda()
    B.kfx_gemm_exact(levels, M, N, K, -0.5, torch.from_numpy(A).cuda(), K, torch.from_numpy(Bm).cuda(), K, 2.0, 3.0,
                     C, N)
    got = C.cpu().numpy()
    bound = 2.0 ** (5 - 8 * levels) * K * np.abs(A).max(1)[:, None] * np.abs(Bm).max(1)[None, :] * 0.5
    err = np.abs(got - ref)
    print(f"levels {levels}: max error / bound = {(err / bound).max():.3f}")
    assert np.all(err <= bound + 4 * np.spacing(np.abs(ref)))


def test_exact_product_float32_operands():
    rng = np.random.default_rng(3)
    M, N, K = 150, 90, 260
    A = rng.standard_normal((M, K)).astype(np.float32)
    Bm = rng.standard_normal((N, K)).astype(np.float32)
    ref, _, _ = exact_sliced_product(A.astype(np.float64), Bm.astype(np.float64), 7)
    C = torch.zeros(M, N, dtype=torch.float64, device="cuda")
    B.kfx_gemm_exact(7, M, N, K, 1.0, torch.from_numpy(A).cuda(), K, torch.from_numpy(Bm).cuda(), K, 0.0, 0.0, C, N)
    assert np.abs(C.cpu().numpy() - ref).max() <= 1e-13 * np.abs(ref).max()


def spd32(n, cond, seed):
    """float32 SPD matrix with eigenvalues spread geometrically over [1/cond, 1] (the range of a
    smoother prediction P_{t+1|t} = P_{t|t} + Q with Q = 1e-2 I and P0 = I has cond <= ~100)."""
    rng = np.random.default_rng(seed)
    Qm, _ = np.linalg.qr(rng.standard_normal((n, n)))
    A = (Qm * np.geomspace(1.0 / cond, 1.0, n)) @ Qm.T
    A = 0.5 * (A + A.T)
    return A.astype(np.float32)


@pytest.mark.parametrize("n,cond", [(257, 100.0), (1024, 100.0), (2048, 100.0), (4096, 100.0), (1024, 1000.0)])
def test_refined_inverse_is_float64_accurate(n, cond):
    A = spd32(n, cond, n)
    dA = torch.from_numpy(A).cuda()
    # float64 CUDA-core reference: Cholesky + two triangular solves with B = I
    A64 = torch.from_numpy(A.astype(np.float64)).cuda()
    X64 = torch.eye(n, dtype=torch.float64, device="cuda")
    st, _ = B.kfx_posv_right(0, n, A64, n, n, X64, n)
    assert st == 0
    X64 = X64.cpu().numpy()
    Xnp = np.linalg.inv(A.astype(np.float64))
    assert np.linalg.norm(X64 - Xnp) <= 1e-12 * np.linalg.norm(Xnp) * cond / 100
    errs = {}
    for mode in (1, 2):
        X = torch.zeros(n, n, dtype=torch.float64, device="cuda")
        st, fi = B.kfx_spd_inverse(mode, n, dA, n, X, n)
        assert st == 0 and fi == -1
        Xg = X.cpu().numpy()
        errs[mode] = np.linalg.norm(Xg - X64) / np.linalg.norm(X64)
    print(f"n {n} cond {cond:g}: float32-class {errs[1]:.2e}, refined {errs[2]:.2e} (vs float64 solve)")
    assert errs[1] <= 1e-3
    assert errs[2] <= 1e-12 * cond / 100


def test_refined_inverse_reports_not_pd():
    n = 300
    A = spd32(n, 50.0, 1).astype(np.float64)
    A[150, :] = 0.0
    A[:, 150] = 0.0
    X = torch.zeros(n, n, dtype=torch.float64, device="cuda")
    st, fi = B.kfx_spd_inverse(2, n, torch.from_numpy(A.astype(np.float32)).cuda(), n, X, n)
    assert st == B.KF_ERR_NOT_PD and fi == 150


def test_exact_product_non_finite_rows_give_nan():
    """A NaN or infinity in a row of A makes that output row NaN (and no other)."""
    rng = np.random.default_rng(11)
    M, N, K = 40, 30, 50
    A = rng.standard_normal((M, K))
    Bm = rng.standard_normal((N, K))
    A[3, 7] = np.nan
    A[9, 0] = np.inf
    C = torch.zeros(M, N, dtype=torch.float64, device="cuda")
    B.kfx_gemm_exact(5, M, N, K, 1.0, torch.from_numpy(A).cuda(), K, torch.from_numpy(Bm).cuda(), K, 0.0, 0.0, C, N)
    got = C.cpu().numpy()
    bad = np.zeros(M, bool)
    bad[[3, 9]] = True
    assert np.all(np.isnan(got[bad])) and np.all(np.isfinite(got[~bad]))


def test_exact_product_wait_limit_timeout_then_recovery():
    """Failure detection of the exact-slice pipeline without a fault: with the pipeline waits
    limited to 1 ns the gate, MMA, TMA and epilogue roles stop at their first unmet wait, the
    kernel waits for what it already issued, frees its tensor memory and the entry point returns
    KF_ERR_TIMEOUT; with the default limit restored the same call matches the scheme."""
    rng = np.random.default_rng(11)
    M, N, K = 256, 128, 2048
    A = rng.standard_normal((M, K))
    Bm = rng.standard_normal((N, K))
    dA, dB = torch.from_numpy(A).cuda(), torch.from_numpy(Bm).cuda()
    C = torch.zeros(M, N, dtype=torch.float64, device="cuda")
    prev = B.kfx_tc_wait_limit(1)
    try:
        for _ in range(2):
            with pytest.raises(B.KfError) as e:
                B.kfx_gemm_exact(7, M, N, K, 1.0, dA, K, dB, K, 0.0, 0.0, C, N)
            assert e.value.status == B.KF_ERR_TIMEOUT
    finally:
        B.kfx_tc_wait_limit(0)
    assert prev == 2_000_000_000
    B.kfx_gemm_exact(7, M, N, K, 1.0, dA, K, dB, K, 0.0, 0.0, C, N)
    ref, ea, eb = exact_sliced_product(A, Bm, 7)
    scale = np.ldexp(1.0, (ea[:, None] + eb[None, :]).astype(np.int64))
    assert np.all(np.abs(C.cpu().numpy() - ref) <= 2.0 ** -50 * scale + 4 * np.spacing(np.abs(ref)))


@pytest.mark.parametrize("levels,K", [(5, 32768), (5, 32769), (6, 4096), (7, 8192)])
def test_exact_product_largest_sums(levels, K):
    """Same-sign rows of the largest digits: the fixed-point sums reach their largest magnitude on both
    sides of the K up to which one 64-bit sum holds all levels; random rows beside them."""
    rng = np.random.default_rng(levels + K)
    M, N = 5, 3
    A = rng.standard_normal((M, K))
    Bm = rng.standard_normal((N, K))
    A[0] = 1.0 - 2.0 ** -50
    A[1] = -(1.0 - 2.0 ** -50)
    Bm[0] = 1.0 - 2.0 ** -50
    ref, ea, eb = exact_sliced_product(A, Bm, levels)
    C = torch.zeros(M, N, dtype=torch.float64, device="cuda")
    B.kfx_gemm_exact(levels, M, N, K, 1.0, torch.from_numpy(A).cuda(), K, torch.from_numpy(Bm).cuda(), K, 0.0, 0.0,
                     C, N)
    # the sums are exact integers, scaled with one rounding
    assert np.array_equal(C.cpu().numpy(), ref)


@pytest.mark.parametrize("alpha,beta,delta", [(1.0, 1.0, 0.0), (-1.0, 1.0, 0.0), (-1.0, 0.0, 1.0), (0.5, -2.0, 0.25)])
@pytest.mark.parametrize("M,N", [(128, 64), (129, 65), (300, 200), (40, 400)])
def test_exact_product_epilogue_forms(alpha, beta, delta, M, N):
    """The epilogue's own loops for unit alpha and beta and its general one, on tiles with and without
    diagonal elements and with ragged edges: the same product plus the same float64 operations."""
    rng = np.random.default_rng(M + N)
    K, levels = 90, 5
    A, Bm, C0 = rng.standard_normal((M, K)), rng.standard_normal((N, K)), rng.standard_normal((M, N))
    dA, dB = torch.from_numpy(A).cuda(), torch.from_numpy(Bm).cuda()
    P = torch.zeros(M, N, dtype=torch.float64, device="cuda")
    B.kfx_gemm_exact(levels, M, N, K, 1.0, dA, K, dB, K, 0.0, 0.0, P, N)
    C = torch.from_numpy(C0.copy()).cuda()
    B.kfx_gemm_exact(levels, M, N, K, alpha, dA, K, dB, K, beta, delta, C, N)
    ref = alpha * P.cpu().numpy()
    if beta != 0.0:
        ref = ref + beta * C0
    ref += delta * np.eye(M, N)
    assert np.allclose(C.cpu().numpy(), ref, rtol=4e-16, atol=4e-16 * np.abs(ref).max())  # fused or not


@pytest.mark.parametrize("N,m", [(512, 64), (640, 40), (1100, 130)])
def test_filter_products_split_over_k(N, m):
    """U^T = P H^T with few output tiles is split over K into integer sums: the mixed filter against the
    oracle at sizes with two and more splits.  Tolerance: the product's bound 2^-35 K on diag P, and the
    mixed path's 1e-4 on means; a lost or doubled split is an error of order one."""
    from paper_1107_4192_gb300 import solver, synth
    from tests.helpers import diag_of, rel_err_elementwise, rel_err_per_step, run_oracle
    prob = synth.mesh_problem(N, m, 3, seed=N)
    out = solver.run(prob, prec=B.KF_PREC_MIXED_BF16X3, solve_prec=B.KF_SOLVE_FP64_MEAN, joseph_every=2)
    ref = run_oracle(prob)
    assert rel_err_elementwise(out["diagP_filt"], diag_of(ref["P_filt"])) <= 2.0 ** -35 * N
    assert rel_err_per_step(out["x_filt"], ref["x_filt"]) <= 1e-4


@pytest.mark.parametrize("f32", [False, True])
@pytest.mark.parametrize("K", [8, 250, 257, 500, 513, 2049, 4100, 6145, 10240, 10241])
def test_slicing_row_lengths(f32, K):
    """Every way a row is held while it is sliced (a warp or a block per row, one to five parts, two passes),
    at the edges of their lengths, with an operand whose leading dimension breaks the 16-byte alignment."""
    rng = np.random.default_rng(K)
    M, N, lda = 9, 3, K + 1
    A = np.zeros((M, lda))
    A[:, :K] = rng.standard_normal((M, K)) * np.exp(rng.uniform(-30, 30, (M, 1)))
    A[2] = 0.0
    A[3, 1:] = 0.0
    Bm = rng.standard_normal((N, K))
    if f32:
        A = A.astype(np.float32)
    dA = torch.from_numpy(A).cuda()
    C = torch.zeros(M, N, dtype=torch.float64, device="cuda")
    B.kfx_gemm_exact(6, M, N, K, 1.0, dA, lda, torch.from_numpy(Bm).cuda(), K, 0.0, 0.0, C, N)
    ref, ea, eb = exact_sliced_product(A[:, :K].astype(np.float64), Bm, 6)
    assert np.array_equal(C.cpu().numpy(), ref)  # digits, sums and one rounding are exact
    A[4, K // 2] = np.inf
    A[5, K - 1] = np.nan
    C.zero_()
    B.kfx_gemm_exact(6, M, N, K, 1.0, torch.from_numpy(A).cuda(), lda, torch.from_numpy(Bm).cuda(), K, 0.0, 0.0, C, N)
    got = C.cpu().numpy()
    bad = np.isin(np.arange(M), [4, 5])
    assert np.all(np.isnan(got[bad])) and np.array_equal(got[~bad], ref[~bad])


@pytest.mark.parametrize("n", [1, 2, 63, 129, 200, 385])
def test_refined_inverse_ragged_sizes(n):
    """The Newton steps on rounded iterates at ragged sizes, against numpy in float64: no worse than the
    conditioning times float64 rounding (cond 100; the bound of the larger sizes' test)."""
    A = spd32(n, 100.0 if n > 1 else 1.0, n)
    X = torch.zeros(n, n, dtype=torch.float64, device="cuda")
    st, fi = B.kfx_spd_inverse(2, n, torch.from_numpy(A).cuda(), n, X, n)
    assert st == 0 and fi == -1
    ref = np.linalg.inv(A.astype(np.float64))
    assert np.linalg.norm(X.cpu().numpy() - ref) <= 1e-12 * np.linalg.norm(ref)
    assert torch.equal(X, X.T)


@pytest.mark.parametrize("n,bad", [(1, (0,)), (31, (30,)), (32, (0, 31)), (33, (32,)), (64, (31, 32)), (65, (64,)),
                                   (1024, (500,)), (1535, (1534,)), (1536, (767,)), (1537, (895, 896, 1536))])
def test_one_launch_factor_and_inverse(n, bad):
    """The float32 factor and triangular inverse around its 32-wide tiles and at the size above which it runs on
    halves: X = W^T W against numpy (float32 sums of 32 terms, 32 x 6e-8 x cond 100 = 2e-4), and the index of the
    first bad pivot (a zero row and column) in either half."""
    A = spd32(n, 100.0 if n > 1 else 1.0, n)
    X = torch.zeros(n, n, dtype=torch.float64, device="cuda")
    for i in bad:
        Z = A.copy()
        Z[i, :] = 0.0
        Z[:, i] = 0.0
        assert B.kfx_spd_inverse(1, n, torch.from_numpy(Z).cuda(), n, X, n) == (B.KF_ERR_NOT_PD, i)
    assert B.kfx_spd_inverse(1, n, torch.from_numpy(A).cuda(), n, X, n) == (0, -1)
    ref = np.linalg.inv(A.astype(np.float64))
    assert np.linalg.norm(X.cpu().numpy() - ref) <= 2e-4 * np.linalg.norm(ref)
