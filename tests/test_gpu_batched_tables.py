"""Plans with entry tables: which instances come from a table and that the others
get what a plan without tables gives them."""
import os

import pytest

import paper_2502_00356_gb300 as bk
from paper_2502_00356_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

WEIGHTS = os.path.join(os.path.dirname(os.path.abspath(bk.__file__)), "weights", "window_mlp.bkw")


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    bk.build()
    return torch.device("cuda:0")


@pytest.fixture(scope="module")
def forms(dev):
    net = bk.LearnedWindow(path=WEIGHTS)
    return {"f64": lambda **k: bk.make_opts(**k), "f32": lambda **k: bk.make_opts(compute=bk.BK_F32, **k),
            "learned": lambda **k: bk.make_opts(learned=net, **k)}


def item(n, seed, params, dtype, dev):
    L = torch.as_tensor(inputs.morton_sorted(inputs.jittered_grid(n, seed=seed)), device=dev)
    return (L, *params, torch.full((n, n), float("nan"), dtype=dtype, device=dev))


def run(items, opts, dtype, chunk=None):
    plan = bk.BatchedPlan([i[0].shape[1] for i in items], dtype=dtype, opts=opts)
    bk.bk_matern_batched(bk.make_descs(items), plan)
    torch.cuda.synchronize()
    return plan


@pytest.mark.parametrize("form", ["f64", "f32", "learned"])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_instances_without_a_table_keep_their_form(dev, forms, form, dtype):
    """Small instances, orders outside the tables' domain (one of them the first and one
    the last of the batch) and a descriptor that does not match, among instances with
    tables: the former bit for bit as the per-entry kernel of the same form gives them
    (a plan with counters has no tables), the latter within twice the forms' bounds."""
    spec = [(600, (1.0, 0.1, 11.0)), (2500, (1.2, 0.1, 0.8)), (40, (1.0, 0.1, 0.5)), (255, (0.7, 0.2, 1.1)), (2100, (0.5, 0.05, 2.3)),
            (1, (2.0, 0.1, 1.0)), (1500, (1.0, 0.1, 0.01)), (700, (1.0, 0.02, 1.5)), (800, (1.0, 0.2, 15.0))]
    opts = forms[form]
    items = [item(n, 30 + k, p, dtype, dev) for k, (n, p) in enumerate(spec)]
    wrong = item(300, 50, (1.0, 0.1, 1.0), dtype, dev)
    ctr = torch.zeros(bk.BK_NUM_COUNTERS, dtype=torch.int64, device=dev)
    refs = [(*i[:4], torch.full_like(i[4], float("nan"))) for i in items]
    run(refs, opts(counters=ctr), dtype)
    plan = bk.BatchedPlan([n for n, _ in spec] + [310], dtype=dtype, opts=opts())
    descs = bk.make_descs(items + [wrong])
    for _ in range(2):  # the second call finds the plan's counters and tables as the first left them
        for i in items:
            i[4].fill_(float("nan"))
        bk.bk_matern_batched(descs, plan)
        torch.cuda.synchronize()
        for (n, p), i, r in zip(spec, items, refs):
            if n < 256 or not 0.02 <= p[2] <= 10.0:
                assert torch.equal(i[4], r[4]), (n, p)
            else:
                tol = 4e-13 if form == "f64" and dtype == torch.float64 else 2e-6
                assert bool(((i[4].double() - r[4].double()).abs() <= tol * r[4].double() + 2e-38).all()), (n, p)
        assert bool(torch.isnan(wrong[4]).all())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        bk.bk_matern_batched(descs, plan)
    want = [i[4].clone() for i in items]
    for i in items:
        i[4].fill_(float("nan"))
    g.replay()
    torch.cuda.synchronize()
    assert all(torch.equal(i[4], w) for i, w in zip(items, want))


@pytest.mark.parametrize("form,dtype,sizes,table", [
    ("f64", torch.float64, [725], True), ("f64", torch.float64, [700], False), ("f64", torch.float64, [900, 100], True),
    ("f64", torch.float64, [700, 100, 20], False), ("f32", torch.float32, [900], False), ("f32", torch.float32, [1024], True),
    ("learned", torch.float32, [1000], False), ("learned", torch.float32, [400] * 8, True), ("learned", torch.float32, [1250, 200], False),
    ("learned", torch.float32, [1260, 200], True), ("learned", torch.float64, [1200], False), ("f32", torch.float64, [400] * 40, False),
    ("f32", torch.float64, [1300], True), ("f32", torch.float64, [1600, 300], False),
    ("f32", torch.float64, [1650, 300], True)])
def test_which_batches_have_tables(dev, forms, form, dtype, sizes, table):
    """By the entries that a table serves; the plan's size is that of its tiles of 32."""
    opts = forms[form]
    # x near 1e-2 throughout: the table's values differ from the per-entry ones in some last bit
    items = [item(n, 60 + k, (1.0, 3.0, 0.9), dtype, dev) for k, n in enumerate(sizes)]
    refs = [(*i[:4], torch.full_like(i[4], float("nan"))) for i in items]
    ctr = torch.zeros(bk.BK_NUM_COUNTERS, dtype=torch.int64, device=dev)
    plan = run(items, opts(), dtype)
    assert plan.info()["total_tiles"] == run(refs, opts(counters=ctr), dtype).info()["total_tiles"] == \
        sum(-(-n // 32) * (-(-n // 32) + 1) // 2 for n in sizes)
    assert all(torch.equal(i[4], r[4]) for i, r in zip(items, refs)) == (not table)
