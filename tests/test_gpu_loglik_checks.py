"""What the fixed-point Cholesky behind bk_gaussian_loglik must refuse, and that
its panels give the same bits every time."""
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
