"""The Matern writers that evaluate entries from a per-call table against the
writers that run the quadrature for every entry (which options with counters
select), over the orders, scales, sizes, types and layouts the tables accept."""
import ctypes

import numpy as np
import pytest

import paper_2502_00356_gb300 as bk
from paper_2502_00356_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# The direct forms' own bounds (FP64 entries to ~1e-13, FP32 to ~1e-6), twice over.
TOL = {torch.float64: 4e-13, torch.float32: 2e-6}


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    bk.build()
    return torch.device("cuda:0")


def direct(**kw):
    ctr = torch.zeros(bk.BK_NUM_COUNTERS, dtype=torch.int64, device="cuda")
    return bk.make_opts(counters=ctr, **kw)


def grid(n, seed, dev, scale=1.0, shift=0.0):
    L = inputs.morton_sorted(inputs.jittered_grid(n, seed=seed))
    return torch.as_tensor(L * scale + shift, device=dev)


def check(got, want):
    g, w = got.double(), want.double()
    small = 1e-300 if got.dtype == torch.float64 else 2e-38  # below: underflow of the FP32 forms
    assert bool(((g - w).abs() <= TOL[got.dtype] * w.abs() + small).all()), \
        float(((g - w).abs() / w.abs().clamp_min(small)).max())


@pytest.mark.parametrize("nu", [0.02, 0.3, 0.5, 1.0, 2.3, 5.0, 10.0])
@pytest.mark.parametrize("beta", [0.008, 0.1, 3.0])
@pytest.mark.parametrize("form", ["f64", "f32", "f64 to f32", "f32 to f64"])
def test_equals_the_direct_evaluation(dev, nu, beta, form):
    """x from the smallest spacings (below the tables for beta = 3) to 175
    (beyond them for beta = 0.008); ld > n, a ragged last tile."""
    n, ld = 733, 740
    L = grid(n, 3, dev)
    L[:, 5] = L[:, 700]                       # a coincident pair
    L[:, 11] = L[:, 12] + 1e-9                # and a very near one
    dtype = torch.float64 if form in ("f64", "f32 to f64") else torch.float32
    kw = {"compute": bk.BK_F32 if form in ("f32", "f32 to f64") else bk.BK_F64}
    out = torch.full((n, ld), float("nan"), dtype=dtype, device=dev)
    bk.bk_matern_tile(L, 1.7, beta, nu, out=out, opts=bk.make_opts(**kw))
    if form == "f32 to f64":  # the direct FP32 writer loses the near pair's distance; FP64 is the reference
        kw = {}
    want = bk.bk_matern_tile(L, 1.7, beta, nu, dtype=dtype, opts=direct(**kw))
    torch.cuda.synchronize()
    got = out[:, :n]
    if form == "f32 to f64":
        assert bool(((got - want).abs() <= 2e-6 * want.abs() + 1e-300).all())
    else:
        check(got, want)
    assert torch.equal(got, got.T) and bool(torch.isnan(out[:, n:]).all())
    assert float(got[5, 700]) == float(np.float32(1.7) if dtype == torch.float32 else 1.7)


@pytest.mark.parametrize("scale,shift", [(1.0, -0.5), (1e6, 3e6), (1e-6, 0.0), (1.0, 1e5)])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_coordinates_of_any_scale(dev, scale, shift, dtype):
    """beta in the coordinates' scale; shifted far from the origin, only the
    coordinates' own rounding is left of the distances."""
    L = grid(800, 4, dev, scale, shift)
    got = bk.bk_matern_tile(L, 1.0, 0.1 * scale, 1.3, dtype=dtype)
    want = bk.bk_matern_tile(L, 1.0, 0.1 * scale, 1.3, dtype=dtype,
                             opts=direct(compute=bk.BK_F64 if dtype == torch.float64 else bk.BK_F32))
    torch.cuda.synchronize()
    check(got, want)


@pytest.mark.parametrize("nu", [0.05, 0.49, 0.5, 3.0])
@pytest.mark.parametrize("width", [0.5, 7.9, 8.1, 31.0, 63.0, 65.0, 300.0])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_scattered_points(dev, nu, width, dtype):
    """Unsorted points over 0.5 to 300 beta, so that every tile spans the whole
    set: on both sides of the spans and distances for which a tile's coordinates
    are kept relative to it."""
    g = torch.Generator(device=dev).manual_seed(int(10 * width))
    L = width * torch.rand((2, 740), generator=g, dtype=torch.float64, device=dev) + 17.0
    L[:, :200] = L[:, 200:400] + 0.01 * torch.rand((2, 200), generator=g, dtype=torch.float64, device=dev)
    got = bk.bk_matern_tile(L, 1.0, 1.0, nu, dtype=dtype)
    want = bk.bk_matern_tile(L, 1.0, 1.0, nu, opts=direct(compute=bk.BK_F64))
    torch.cuda.synchronize()
    assert torch.equal(got, got.T)
    check(got, want)


@pytest.mark.parametrize("m,n", [(8192, 64), (63, 9001), (2048, 257), (1, 600000)])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_blocks(dev, m, n, dtype):
    l1, l2 = grid(m, 5, dev), grid(n, 6, dev) * 0.8 + 0.1
    got = bk.bk_matern_tile2(l1, l2, 0.6, 0.15, 1.9, dtype=dtype)
    want = bk.bk_matern_tile2(l1, l2, 0.6, 0.15, 1.9, dtype=dtype,
                              opts=direct(compute=bk.BK_F64 if dtype == torch.float64 else bk.BK_F32))
    torch.cuda.synchronize()
    check(got, want)


@pytest.mark.parametrize("params", [(1.0, 0.1, 10.5), (1.0, 0.1, 0.01), (1.0, 1e-9, 1.5), (1e-25, 0.1, 1.5),
                                    (1e25, 0.1, 1.5), (0.0, 0.1, 1.5), (1.0, 1e9, 1.5)])
def test_outside_the_domain_the_direct_writer_runs(dev, params):
    L = grid(730, 7, dev)
    for dtype in (torch.float64, torch.float32):
        kw = {"compute": bk.BK_F64 if dtype == torch.float64 else bk.BK_F32}
        got = bk.bk_matern_tile(L, *params, dtype=dtype)
        want = bk.bk_matern_tile(L, *params, dtype=dtype, opts=direct(**kw))
        torch.cuda.synchronize()
        bits = torch.int64 if dtype == torch.float64 else torch.int32  # x = 1e9 and more is NaN on both sides
        assert torch.equal(got.view(bits), want.view(bits))


def test_not_finite_locations(dev):
    """NaN and infinite coordinates give what the direct writer gives."""
    L = grid(730, 8, dev)
    L[0, 100], L[1, 300] = float("nan"), float("inf")
    for dtype in (torch.float64, torch.float32):
        got = bk.bk_matern_tile(L, 1.0, 0.1, 1.5, dtype=dtype)
        want = bk.bk_matern_tile(L, 1.0, 0.1, 1.5, dtype=dtype,
                                 opts=direct(compute=bk.BK_F64 if dtype == torch.float64 else bk.BK_F32))
        torch.cuda.synchronize()
        assert torch.equal(torch.isnan(got), torch.isnan(want))
        ok = ~torch.isnan(want)
        check(got[ok], want[ok])


def test_workspace_arguments_and_streams(dev):
    n = 800
    L = grid(n, 9, dev)
    need = bk.lib().bk_matern_workspace(n, n)
    assert bk.lib().bk_matern_workspace(700, 700) == 8 * bk.BK_COSH_TABLE_LEN < need
    work = torch.empty(need + 256, dtype=torch.uint8, device=dev)
    out = torch.empty((n, n), dtype=torch.float64, device=dev)
    call = lambda off, size: bk.lib().bk_matern_tile_ws(
        L.data_ptr(), n, 1.0, 0.1, 1.5, out.data_ptr(), n, bk.BK_F64, None,
        ctypes.c_void_p(work.data_ptr() + off), size, torch.cuda.current_stream().cuda_stream or None)
    assert call(8, need) == bk.BK_ERR_INVALID_ARG
    want = bk.bk_matern_tile(L, 1.0, 0.1, 1.5)
    assert call(0, need) == bk.BK_OK
    torch.cuda.synchronize()
    assert torch.equal(out, want)
    assert call(0, need - 1) == bk.BK_OK  # too small for the table: the direct writer
    torch.cuda.synchronize()
    assert not torch.equal(out, want)
    check(out, want)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    got = [bk.bk_matern_tile(L, 1.0, 0.1, 1.5, stream=s) for _ in range(3)]
    s.synchronize()
    assert all(torch.equal(g, want) for g in got)


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_batched_instances_with_and_without_tables(dev, dtype):
    """Sizes on both sides of the tables' least, and parameters outside their
    domain, in one plan: every instance as a single call gives it."""
    sizes, params = [900, 40, 724, 725, 1300], [(1.0, 0.1, 0.5), (2.0, 0.1, 1.1), (1.0, 0.2, 0.7), (0.5, 0.05, 2.2),
                                                (1.0, 0.1, 12.0)]
    items = [(grid(n, 20 + n, dev), *p, torch.full((n, n), float("nan"), dtype=dtype, device=dev))
             for n, p in zip(sizes, params)]
    plan = bk.BatchedPlan(sizes, dtype=dtype)
    for shape in ("default", "tuned"):
        if shape == "tuned":
            plan.autotune(bk.make_descs(items))
        for it in items:
            it[4].fill_(float("nan"))
        bk.bk_matern_batched(bk.make_descs(items), plan)
        for L, s2, be, nu, out in items:
            want = bk.bk_matern_tile(L, s2, be, nu, dtype=dtype)
            torch.cuda.synchronize()
            check(out, want)
