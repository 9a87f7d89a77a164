"""Minimum-norm calls on a GPU that is nearly full: the slices of the tensor-core products are left out when they do not
fit, and the call needs no more memory than with float64 products throughout."""
from contextlib import contextmanager

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


@contextmanager
def memory_left(leave):
    """Holds all of the GPU's free memory but `leave` bytes."""
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    if free < 2 * leave:
        pytest.skip("the GPU is in use")
    room = torch.empty(free - leave, dtype=torch.uint8, device="cuda")
    try:
        yield
    finally:
        del room
        torch.cuda.empty_cache()


def inputs(N, m, T, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    randn = lambda *s: torch.randn(*s, generator=g, device="cuda", dtype=torch.float64)
    one = torch.ones(1, device="cuda", dtype=torch.float64)
    return randn(m, N), one, one.expand(m).contiguous(), randn(T, m)


def per_source(X, ref):
    return float(((X - ref).norm(dim=0) / ref.norm(dim=0)).max())


def test_mne_solve_without_room_for_slices():
    """H of 1.6 GB, 3 GB left: H C fits, the slices (44 bytes per element) do not."""
    N, m, T = 400_000, 512, 4
    H, C, R, Y = inputs(N, m, T, 1)
    X, ref = torch.empty(2, T, N, dtype=torch.float64, device="cuda")
    B.mne_solve(H, C, 0, R, 1, Y, N, m, T, 1.0, ref)
    with memory_left(3 * 10 ** 9):
        B.mne_solve(H, C, 0, R, 1, Y, N, m, T, 1.0, X)
    assert per_source(X, ref) <= 1e-11


@pytest.mark.parametrize("keep_X", [False, True])
def test_mne_init_without_room_for_slices(keep_X):
    """X and its differences take 0.64 GB each, their slices 1.1 GB more."""
    N, m, T = 20_000, 64, 4000
    H, C, R, Y = inputs(N, m, T, 2)
    x0, Q = torch.empty(N, dtype=torch.float64, device="cuda"), torch.empty(N, N, dtype=torch.float64, device="cuda")
    X = torch.empty(T, N, dtype=torch.float64, device="cuda") if keep_X else None
    B.mne_init(H, C, 0, R, 1, Y, N, m, T, 1.0, X, x0, Q)
    x0_ref, d, part = x0.clone(), Q.diagonal().clone(), Q[:, :500].clone()
    x0.zero_()
    Q.zero_()
    with memory_left((1100 if keep_X else 1700) * 10 ** 6):
        B.mne_init(H, C, 0, R, 1, Y, N, m, T, 1.0, X, x0, Q)
    assert torch.allclose(x0, x0_ref, rtol=1e-11, atol=1e-11 * float(x0_ref.abs().max()))
    s = d.sqrt()
    assert float(((Q[:, :500] - part) / s[:, None] / s[:500]).abs().max()) <= 1e-11
