"""What the fixed-point Cholesky behind bk_gaussian_loglik must refuse, and that
its panels give the same bits every time."""
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


@pytest.mark.parametrize("n,times", [(72, 60), (700, 60), (5003, 6)])
def test_every_run_gives_the_same_bits(dev, n, times):
    """Panels whose solving warps read a diagonal block while one of them stores
    its factor (four warps; five from 4,672 rows on) must not read the factor:
    integer arithmetic in a fixed order then leaves no two results apart."""
    L = torch.as_tensor(inputs.morton_sorted(inputs.jittered_grid(n, seed=4)), device=dev)
    A = bk.bk_matern_tile(L, 1.0, 0.1, 0.5)
    z = torch.randn(n, generator=torch.Generator(device=dev).manual_seed(2), dtype=torch.float64, device=dev)
    first = None
    for _ in range(times):
        a, y = A.clone(), torch.empty_like(z)
        out = bk.bk_gaussian_loglik(a, z, y=y)
        torch.cuda.synchronize()
        got = [t.view(torch.int64) for t in (a, y, out)]
        if first is None:
            first = got
        assert bool(torch.isfinite(out).all()) and all(torch.equal(g, f) for g, f in zip(got, first))


def both(A, dev):
    """(out, failures counted) of the fixed-point path and of the FP64 one."""
    n = A.shape[0]
    res = []
    for fixed in (True, False):
        a, z = A.clone(), torch.ones(n, dtype=torch.float64, device=dev)
        y, out = torch.empty_like(z), torch.empty(3, dtype=torch.float64, device=dev)
        ctr = torch.zeros(bk.BK_NUM_COUNTERS, dtype=torch.int64, device=dev)
        opts = bk.make_opts(counters=ctr)
        if fixed:
            bk.bk_gaussian_loglik(a, z, y=y, out=out, opts=opts)
        else:
            assert bk.lib().bk_gaussian_loglik(a.data_ptr(), n, n, z.data_ptr(), y.data_ptr(), out.data_ptr(), ctypes.byref(opts),
                                               torch.cuda.current_stream().cuda_stream or None) == bk.BK_OK
        torch.cuda.synchronize()
        res.append((out.cpu().numpy(), int(ctr[bk.BK_CTR_FAIL])))
    return res


def refused(A, dev):
    (fixed, count), (plain, _) = both(A, dev)
    assert np.all(np.isnan(plain)), "the FP64 path accepts it"
    assert np.all(np.isnan(fixed)) and count == 1, (fixed, count)


# rows of one group of 8, across groups, across panels (64) and row blocks (128),
# and the small pivot, the twin and the third variable far apart
TRIPLES = [(0, 1, 2), (1, 2, 7), (6, 7, 8), (7, 8, 9), (5, 20, 40), (15, 16, 63), (62, 63, 64), (63, 64, 65), (2, 3, 299),
           (2, 60, 70), (2, 70, 200), (126, 127, 128), (127, 128, 129), (100, 190, 260), (270, 280, 299)]


@pytest.mark.parametrize("i,j,k", TRIPLES)
@pytest.mark.parametrize("gap,entry", [(40, 0.5), (40, 0.25), (20, -0.7), (52, 0.9)])
def test_a_large_entry_below_a_small_pivot(dev, i, j, k, gap, entry):
    """Two variables that nearly coincide and a third correlated with one of
    them only: eigenvalue about -entry^2/2.  L_kj would be entry 2^{gap/2}."""
    A = torch.eye(300, dtype=torch.float64, device=dev)
    A[j, i] = A[i, j] = 1.0
    A[j, j] += 2.0 ** -gap
    A[k, j] = A[j, k] = entry
    refused(A, dev)


@pytest.mark.parametrize("row,columns", [(16, range(16)), (40, range(16)), (63, range(32)), (64, range(16)),
                                         (200, range(64)), (250, range(30, 46)), (299, range(0, 299, 8)),
                                         (1090, range(0, 1088, 68)), (1090, range(0, 1024, 64))])
def test_a_row_longer_than_its_diagonal(dev, row, columns):
    """Entries of 1.99 beside unit diagonals, each within what one entry may be;
    sixteen of them take a 64-bit sum of their squares once around."""
    A = torch.eye(max(row + 10, 300), dtype=torch.float64, device=dev)
    for c in columns:
        A[row, c] = A[c, row] = 1.99
    refused(A, dev)


@pytest.mark.parametrize("n", [24, 130, 300])
def test_random_indefinite_matrices_with_a_nearly_singular_block(dev, n):
    """Correlation matrices of nearly coinciding variables, one entry moved so
    that the smallest eigenvalue is clearly negative."""
    rng = np.random.default_rng(n)
    for _ in range(12):
        B = rng.standard_normal((n, max(2, n // 4)))
        A = B @ B.T + 10.0 ** -rng.uniform(2, 11) * np.eye(n)
        d = np.sqrt(np.diag(A)) * 2.0 ** rng.uniform(-1, 1, n)
        A = A / d[:, None] / d[None, :]
        i, j = sorted(rng.choice(n, 2, replace=False))
        A[i, j] = A[j, i] = A[i, j] + rng.choice([-1, 1]) * rng.uniform(0.05, 0.4)
        assert np.linalg.eigvalsh(A)[0] < -1e-3
        refused(torch.as_tensor(A, device=dev), dev)


def test_rows_at_the_end_of_their_scale_pass(dev):
    """Diagonals just below a power of four, correlations up to 1 - 2^-30: what
    the tests above refuse must not refuse these."""
    n = 200
    g = torch.Generator(device=dev).manual_seed(5)
    u = torch.rand(n, generator=g, dtype=torch.float64, device=dev) * 2.0 ** -15
    d = 2.0 - 2.0 ** -51 - torch.randint(0, 2, (n,), generator=g, device=dev) * 0.5
    A = torch.exp(-(u[:, None] - u[None, :]).abs()) * d[:, None] * d[None, :]
    A += torch.diag(torch.full((n,), 2.0 ** -32, dtype=torch.float64, device=dev))
    A = torch.minimum(A, torch.full_like(A, 4.0 - 2.0 ** -50))
    (fixed, count), (plain, _) = both(A, dev)
    # condition about 2^40: the two log determinants agree to n 2^-53 of that per pivot
    assert count == 0 and abs(fixed[1] - plain[1]) <= 1e-2 * n


def test_small_entries_of_the_factor_by_the_fp64_factorisation(dev):
    """A = L L^T with entries of 2^-70 below a unit diagonal: in fixed point (60
    fraction bits) they are lost, with fp64=True the factor has them exactly."""
    n = 130
    A = torch.eye(n, dtype=torch.float64, device=dev)
    for i, j in ((5, 1), (70, 3), (129, 64), (128, 127)):
        A[i, j] = A[j, i] = 2.0 ** -70
    z = torch.ones(n, dtype=torch.float64, device=dev)
    a, b = A.clone(), A.clone()
    out, plain = bk.bk_gaussian_loglik(a, z), bk.bk_gaussian_loglik(b, z, fp64=True)
    torch.cuda.synchronize()
    assert torch.equal(out, plain) and torch.equal(b, A) and float((a - A).abs().max()) <= 2.0 ** -59
