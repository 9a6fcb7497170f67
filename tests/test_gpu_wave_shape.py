"""Launch shapes of the sorted evaluation kernels (blocks of four to eight warps,
one or several rounds) and the gradient's two node loops, at the edges of their
ranges: results depend on neither the other pairs of a call nor its size."""
import numpy as np
import pytest

import oracle
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


@pytest.mark.parametrize("warps,extra", [(1, 0), (4, 1), (8, 0), (8, 1), (12, 1), (16, 0), (16, 1), (17, 0),
                                         (20, 1), (21, -7), (24, 0), (24, 1), (31, 5), (48, 1)])
def test_any_number_of_warps_an_sm(dev, warps, extra):
    """`warps` runs of 32 pairs an SM and a few more or less, against calls of 1,000.
    A pair's arithmetic may differ in the last bits only (a warp's vote on the
    series of 2 cosh h)."""
    n = 32 * torch.cuda.get_device_properties(dev).multi_processor_count * warps + extra
    x, nu = (torch.as_tensor(a, device=dev) for a in inputs.kv_pairs(n, seed=warps, nu_hi=10.0))
    k = bk.bk_eval(x, nu)
    g = bk.bk_eval_grad(x, nu)
    for i in (0, n // 2, max(0, n - 1000)):
        xs, ns = x[i:i + 1000].contiguous(), nu[i:i + 1000].contiguous()
        part = [bk.bk_eval(xs, ns), *bk.bk_eval_grad(xs, ns)]
        torch.cuda.synchronize()
        for whole, p in zip((k, *g), part):
            w = whole[i:i + 1000]
            # (dK/dnu, a difference, relative to K and itself)
            assert bool(((w - p).abs() <= 1e-13 * torch.maximum(p.abs(), part[0])).all())


def test_gradient_node_loops(dev):
    """Orders from 0 and tiny (1 - e^{-2 nu t} in fixed point) to windows that start
    off zero, arguments on both sides of the uncentred loop's range (x cosh t1
    below 690)."""
    X, V = (a.ravel() for a in np.meshgrid([1e-3, 0.01, 0.3, 2.0, 30.0, 300.0, 500.0, 600.0, 640.0, 680.0],
                                           [0.0, 1e-14, 1e-9, 1e-5, 0.01, 0.5, 7.0, 19.0, 20.0]))
    k, dx, dn = (t.cpu().numpy() for t in bk.bk_eval_grad(torch.as_tensor(X, device=dev),
                                                          torch.as_tensor(V, device=dev)))
    wk, wx, wn = oracle.besselk_grad(X, V)
    tiny = (V > 0.0) & (V < 1e-6)  # the oracle's difference has no digits there: linear in nu
    wn[tiny] = V[tiny] / 1e-5 * oracle.besselk_grad(X[tiny], np.full(tiny.sum(), 1e-5))[2]
    assert np.abs(k / wk - 1).max() <= 1e-10 and np.abs(dx / wx - 1).max() <= 1e-10
    assert (np.abs(dn - wn) / np.maximum(np.abs(wn), wk)).max() <= 1e-10
    assert np.all(dn[V == 0.0] == 0.0)
    small = (V > 1e-10) & (V < 0.1)  # (below, 1 - e^{-2 nu h} itself is lost to rounding)
    assert np.abs(dn[small] / wn[small] - 1).max() <= 1e-4
