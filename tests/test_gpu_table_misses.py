"""Entries that an entry table does not hold: far pairs (evaluated with the plain
form's e^{-2 nu h}, or zero where they underflow), coincident ones, values at
the lower end of FP32."""
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


def grid(n, seed, dev, scale=1.0):
    return torch.as_tensor(inputs.morton_sorted(inputs.jittered_grid(n, seed=seed)) * scale, device=dev)


def direct(**kw):
    """Options that ask for the per-entry evaluation."""
    return bk.make_opts(counters=torch.zeros(bk.BK_NUM_COUNTERS, dtype=torch.int64, device="cuda"), **kw)


@pytest.mark.parametrize("nu", [0.02, 0.5, 2.3, 10.0])
@pytest.mark.parametrize("width", [150.0, 700.0, 2000.0, 40000.0])
@pytest.mark.parametrize("block", [False, True])
def test_far_pairs(dev, nu, width, block):
    """x up to `width` and beyond: the tables end at 90, FP64 underflows past 745,
    FP32 past 104.  Twice the direct forms' bounds (1e-13, 1e-6), and an ulp of
    the smallest numbers."""
    n = 760
    L, M = grid(n, 1, dev, width), grid(900, 2, dev, width)
    for dtype, compute in ((torch.float64, bk.BK_F64), (torch.float32, bk.BK_F64), (torch.float32, bk.BK_F32)):
        call = (lambda o: bk.bk_matern_tile2(L, M, 1.5, 1.0, nu, dtype=dtype, opts=o)) if block else \
               (lambda o: bk.bk_matern_tile(L, 1.5, 1.0, nu, dtype=dtype, opts=o))
        got, want = call(bk.make_opts(compute=compute)).double(), call(direct(compute=compute)).double()
        torch.cuda.synchronize()
        small = 1e-300 if dtype == torch.float64 else 2e-38
        tol = 4e-13 if dtype == torch.float64 else 2e-6 if compute == bk.BK_F32 else 2.0 ** -23
        assert bool(((got - want).abs() <= tol * want.abs() + small).all())
        assert bool((got >= 0).all())


def test_every_path_to_an_entry_in_one_matrix(dev):
    """Coincident, near, tabulated, far and underflowing pairs side by side, more
    points than the scan of the distances takes (8,192): the table is complete."""
    n = 9000
    L = torch.cat([grid(4000, 3, dev, 1.0), grid(3000, 4, dev, 1e-3) + 5.0, grid(2000, 5, dev, 3000.0)], dim=1)
    L[:, 8990:] = L[:, :10]
    L = L.contiguous()
    got, want = (bk.bk_matern_tile(L, 0.7, 1.0, 1.2, opts=o) for o in (None, direct()))
    torch.cuda.synchronize()
    assert bool(((got - want).abs() <= 4e-13 * want.abs() + 1e-300).all())
    assert bool((got.diagonal() == 0.7).all()) and float(got[0, 8990]) == 0.7


@pytest.mark.parametrize("sigma2,width", [(1e-20, 62.0), (1e-20, 70.0), (1e-10, 75.0), (1.0, 100.0), (1e-20, 45.0)])
def test_no_fp32_entry_is_negative(dev, sigma2, width):
    """Down to where FP32 ends (2^-149) a covariance is never below zero, and the
    subnormal ones are within a few of their units of the FP64 values."""
    L, M = grid(2500, 6, dev, width), grid(1700, 7, dev, width)
    for nu in (0.3, 1.5, 7.0):
        for got, want in ((bk.bk_matern_tile(L, sigma2, 1.0, nu, dtype=torch.float32), bk.bk_matern_tile(L, sigma2, 1.0, nu)),
                          (bk.bk_matern_tile2(L, M, sigma2, 1.0, nu, dtype=torch.float32),
                           bk.bk_matern_tile2(L, M, sigma2, 1.0, nu))):
            torch.cuda.synchronize()
            assert bool((got >= 0).all()), float(got.min())
            low = want < 2.0 ** -130
            assert bool(low.any()) and float((got.double() - want)[low].abs().max()) <= 2.0 ** -130 * 2e-6 + 64 * 2.0 ** -149


@pytest.mark.parametrize("n,pad", [(725, 0), (733, 4), (800, 0), (850, 0), (961, 7), (1343, 0), (1345, 0), (1450, 1), (1537, 7)])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_a_matrix_is_the_same_in_host_memory(dev, n, pad, dtype):
    """Halves of tiles, or whole ones (columns that do not start on 32 bytes, from
    n = 1,345 on), where a matrix in device memory takes quarters."""
    L = inputs.morton_sorted(inputs.jittered_grid(n, seed=8))
    want = bk.bk_matern_tile(torch.as_tensor(L, device=dev), 0.9, 0.1, 1.3, dtype=dtype)
    got = torch.full((n, n + pad), -1.0, dtype=dtype, pin_memory=True)
    work = torch.empty(bk.matern_tile_host_workspace(n, dtype, staged=False), dtype=torch.uint8, device=dev)
    bk.bk_matern_tile_host(torch.as_tensor(L).pin_memory(), 0.9, 0.1, 1.3, got, work)
    torch.cuda.synchronize()
    assert torch.equal(got[:, :n], want.cpu()) and bool((got[:, n:] == -1.0).all())


@pytest.mark.parametrize("sigma2,table", [(2.0 ** 50, True), (2.0 ** 50 * 1.001, False), (1e19, False)])
def test_fp32_tables_hold_values_up_to_2_to_the_50(dev, sigma2, table):
    """A larger sigma^2 takes the writer without a table, which leaves the scratch as
    it was, instead of a table whose records near x = 0 hold nothing."""
    n = 800
    L = grid(n, 9, dev)
    out = torch.empty((n, n), dtype=torch.float32, device=dev)
    work = torch.full((bk.lib().bk_matern_workspace(n, n),), 0xA5, dtype=torch.uint8, device=dev)
    assert bk.lib().bk_matern_tile_ws(L.data_ptr(), n, sigma2, 0.1, 1.5, out.data_ptr(), n, bk.BK_F32, None, work.data_ptr(),
                                      work.numel(), torch.cuda.current_stream().cuda_stream or None) == bk.BK_OK
    want = bk.bk_matern_tile(L, sigma2, 0.1, 1.5, opts=direct())
    torch.cuda.synchronize()
    assert bool((work != 0xA5).any()) == table
    assert bool(((out.double() - want).abs() <= 2e-6 * want).all())


def test_two_sets_that_start_at_the_same_address(dev):
    """m and n points from one buffer: x and y of the second set are other parts of
    it, and its distances reach further than the first set's."""
    m, n = 1000, 700
    g = torch.Generator(device=dev).manual_seed(3)
    buf = torch.rand(2 * m, generator=g, dtype=torch.float64, device=dev)
    buf[m:] += 10.0  # the first set lies in [0, 1] x [10, 11], the second's y also in [0, 1]
    out = torch.empty((n, m), dtype=torch.float64, device=dev)
    work = torch.zeros(bk.lib().bk_matern_workspace(m, n), dtype=torch.uint8, device=dev)
    assert bk.lib().bk_matern_tile2_ws(buf.data_ptr(), m, buf.data_ptr(), n, 1.0, 1.0, 1.5, out.data_ptr(), m, bk.BK_F64, None,
                                       work.data_ptr(), work.numel(), torch.cuda.current_stream().cuda_stream or None) == bk.BK_OK
    want = bk.bk_matern_tile2(buf.view(2, m), buf[:2 * n].view(2, n).clone(), 1.0, 1.0, 1.5, opts=direct())
    torch.cuda.synchronize()
    assert bool(((out - want).abs() <= 4e-13 * want).all())
