"""Buffers that the binding allocates for a call on another stream than the
current one: never a block that the current stream may still be working on."""
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


@pytest.mark.parametrize("kind", ["torch", "int", "default"])
def test_scratch_for_another_stream_is_no_block_of_the_current_one(dev, kind):
    """A block freed on the current stream goes to its next scratch, and to
    nothing on another stream (no kernel runs here)."""
    current, other = torch.cuda.Stream(), torch.cuda.Stream()
    target = {"torch": other, "int": other.cuda_stream, "default": 0}[kind]
    nbytes = 37 << 20
    with torch.cuda.stream(current):
        t = bk._scratch(nbytes, dev, None)
        p = t.data_ptr()
        del t
        there = bk._scratch(nbytes, dev, target)
        outputs = bk._empty((nbytes // 8,), torch.float64, dev, target)
        here = bk._scratch(nbytes, dev, None)
        assert there.data_ptr() != p and outputs.data_ptr() != p and here.data_ptr() == p
    torch.cuda.synchronize()


def test_interleaved_calls_on_two_streams(dev):
    """Calls of the current stream and of another in turn, with no wait between
    them: each gives what it gives alone."""
    ns = (1500, 1100)
    locs = [torch.as_tensor(inputs.morton_sorted(inputs.jittered_grid(n, seed=n)), device=dev) for n in ns]
    params = [(1.0, 0.1, 1.3), (0.7, 0.05, 0.6)]
    want = [bk.bk_matern_tile(L, *p) for L, p in zip(locs, params)]
    zs = [torch.ones(n, dtype=torch.float64, device=dev) for n in ns]
    lik = [bk.bk_gaussian_loglik(w.clone(), z) for w, z in zip(want, zs)]
    outs = [[torch.empty_like(w) for w in want] for _ in range(8)]
    liks = [[torch.empty(3, dtype=torch.float64, device=dev) for _ in ns] for _ in outs]
    ys = [[torch.empty_like(z) for z in zs] for _ in outs]
    other = torch.cuda.Stream()
    torch.cuda.synchronize()
    for o, l, y in zip(outs, liks, ys):
        for k, stream in enumerate((None, other)):
            bk.bk_matern_tile(locs[k], *params[k], out=o[k], stream=stream)
        for k, stream in enumerate((None, other)):
            bk.bk_gaussian_loglik(o[k], zs[k], y=y[k], out=l[k], stream=stream)
    torch.cuda.synchronize()
    for o, l in zip(outs, liks):
        for k in range(2):
            assert torch.equal(l[k], lik[k])
            assert torch.equal(o[k].tril(-1), want[k].tril(-1))  # what the factor leaves of the matrix
