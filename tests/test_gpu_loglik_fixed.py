"""The fixed-point Cholesky behind bk_gaussian_loglik_ws against the FP64 one
behind bk_gaussian_loglik (no workspace), at the edges of its panels (64), row
blocks (128) and tiles, with badly scaled rows, and on matrices that are not
positive definite."""
import ctypes

import numpy as np
import pytest

import paper_2502_00356_gb300 as bk
from paper_2502_00356_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    bk.build()
    return torch.device("cuda:0")


def fp64_path(a, z, opts=None):
    n, ld = a.shape
    y, out = torch.empty_like(z), torch.empty(3, dtype=torch.float64, device=a.device)
    rc = bk.lib().bk_gaussian_loglik(a.data_ptr(), n, ld, z.data_ptr(), y.data_ptr(), out.data_ptr(), None,
                                     torch.cuda.current_stream().cuda_stream or None)
    assert rc == bk.BK_OK
    return y, out


@pytest.mark.parametrize("n", [1, 2, 63, 64, 65, 96, 97, 127, 128, 129, 191, 192, 193, 257, 705])
@pytest.mark.parametrize("spread", [0, 12])
def test_equals_the_fp64_factorisation(dev, n, spread):
    """Random A = B B^T/n + I (condition below 10), rows scaled by 10^U(-spread,
    spread).  Both factorisations err by at most about n 2^-53 of a row's norm
    per entry; they agree to 16 times that."""
    g = torch.Generator(device=dev).manual_seed(n)
    B = torch.randn((n, n), generator=g, dtype=torch.float64, device=dev)
    d = 10.0 ** (spread * (2 * torch.rand(n, generator=g, dtype=torch.float64, device=dev) - 1))
    A = (B @ B.T / n + torch.eye(n, dtype=torch.float64, device=dev)) * d[:, None] * d[None, :]
    z = d * torch.randn(n, generator=g, dtype=torch.float64, device=dev)
    tol = 16 * n * 2.0 ** -53
    ld = n + 5
    a = torch.full((n, ld), 7.0, dtype=torch.float64, device=dev)
    a[:, :n] = A
    ref = a.clone()
    y = torch.empty_like(z)
    out = bk.bk_gaussian_loglik(a, z, y=y)
    yr, outr = fp64_path(ref, z)
    torch.cuda.synchronize()
    L, R = a[:, :n].T.tril(), ref[:, :n].T.tril()
    assert float(((L - R) / d[:, None]).abs().max()) <= 4 * tol  # row norms are below 3 d
    assert float((y - yr).abs().max()) <= 16 * tol * max(1.0, float(yr.abs().max()))
    assert float((out - outr).abs().max()) <= 16 * tol * max(float(n), float(outr.abs().max()))
    assert torch.equal(a[:, :n].tril(-1), A.tril(-1)) and bool((a[:, n:] == 7.0).all())


def test_several_tiles_a_block(dev):
    """n = 3,001: rows of tiles longer than a block's share, a ragged last panel."""
    n = 3001
    L = torch.as_tensor(inputs.morton_sorted(inputs.jittered_grid(n, seed=3)), device=dev)
    A = bk.bk_matern_tile(L, 1.0, 0.1, 0.5)
    z = torch.randn(n, generator=torch.Generator(device=dev).manual_seed(1), dtype=torch.float64, device=dev)
    f = torch.linalg.cholesky(A)
    a = A.clone()
    y = torch.empty_like(z)
    out = bk.bk_gaussian_loglik(a, z, y=y)
    torch.cuda.synchronize()
    # condition ~ 1e4: entries agree to that times n 2^-53 at the very most
    assert float((a.T.tril() - f).abs().max()) <= 1e-10
    yr = torch.linalg.solve_triangular(f, z[:, None], upper=False)[:, 0]
    assert float((y - yr).norm() / yr.norm()) <= 1e-10
    assert abs(float(out[1]) - float(2 * f.diagonal().log().sum())) <= 1e-9 * n


@pytest.mark.parametrize("fault", ["late pivot", "large entry", "nan", "inf", "zero diagonal", "first column"])
def test_not_positive_definite(dev, fault):
    n = 300
    A = torch.eye(n, dtype=torch.float64, device=dev)
    if fault == "late pivot":
        A[290, 290] = -1e-9
    elif fault == "large entry":
        A[200, 100] = A[100, 200] = 1.5
    elif fault == "nan":
        A[250, 60] = A[60, 250] = float("nan")
    elif fault == "inf":
        A[130, 130] = float("inf")
    elif fault == "zero diagonal":
        A[64, 64] = 0.0
    else:
        A[5, 0] = A[0, 5] = -3.0
    ctr = torch.zeros(bk.BK_NUM_COUNTERS, dtype=torch.int64, device=dev)
    out = bk.bk_gaussian_loglik(A, torch.ones(n, dtype=torch.float64, device=dev), opts=bk.make_opts(counters=ctr))
    torch.cuda.synchronize()
    assert np.all(np.isnan(out.cpu().numpy())) and int(ctr[bk.BK_CTR_FAIL]) >= 1


@pytest.mark.parametrize("e", [-1070, -1041, -1022, 1000])
def test_scales_at_the_ends_of_the_exponent_range(dev, e):
    """A = 4^{e/2} (I + u), u_10 = 1/2: its factor is exact but for sqrt(3)/2."""
    n = 70
    A = torch.eye(n, dtype=torch.float64, device=dev)
    A[1, 0] = A[0, 1] = 0.5
    A *= 2.0 ** (e // 2)
    A *= 2.0 ** (e - e // 2)
    y = torch.empty(n, dtype=torch.float64, device=dev)
    out = bk.bk_gaussian_loglik(A, torch.zeros(n, dtype=torch.float64, device=dev), y=y)
    torch.cuda.synchronize()
    root = 2.0 ** (e / 2)
    assert abs(float(A[0, 0]) / root - 1) <= 2.0 ** -50 and abs(float(A[0, 1]) / root - 0.5) <= 2.0 ** -50
    assert abs(float(A[1, 1]) / root - 0.75 ** 0.5) <= 2.0 ** -50
    assert abs(float(A[69, 69]) / root - 1) <= 2.0 ** -50
    ld = n * e * np.log(2.0) + np.log(0.75)
    assert abs(float(out[1]) - ld) <= 2.0 ** -45 * abs(ld)


def test_workspace_arguments(dev):
    n = 100
    a = torch.eye(n, dtype=torch.float64, device=dev)
    z, y, out = (torch.ones(n, dtype=torch.float64, device=dev) for _ in range(3))
    need = bk.lib().bk_gaussian_loglik_workspace(n)
    work = torch.empty(need + 256, dtype=torch.uint8, device=dev)
    call = lambda off, size: bk.lib().bk_gaussian_loglik_ws(
        a.data_ptr(), n, n, z.data_ptr(), y.data_ptr(), out.data_ptr(), None, ctypes.c_void_p(work.data_ptr() + off),
        size, torch.cuda.current_stream().cuda_stream or None)
    assert call(8, need) == bk.BK_ERR_INVALID_ARG
    for size in (need, need - 1):  # too small: the FP64 path
        assert call(0, size) == bk.BK_OK
        torch.cuda.synchronize()
        assert float(out[1]) == 0.0 and float(out[2]) == n
