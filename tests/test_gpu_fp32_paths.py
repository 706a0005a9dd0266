"""The FP32 distance tiles and what runs on the pruned lists: list lengths at
the edges of the register layouts, split key ranges, the pruned FP32 tiles
against the unpruned ones, and the per-row recomputation of uncertified
tensor-tile rows. Bit-exact against the oracle or between the paths."""
import numpy as np
import pytest

import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - deselected on CPU runs
    pytest.skip("needs a CUDA device", allow_module_level=True)


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2507_14261_gb300 as P
    return P.Context(0)


def _knn(ctx, X, k, prec, prune):
    ctx.set_knn_pruning(prune)
    nbr, dist = ctx.knn_graph(X, k, prec)
    ctx.set_knn_pruning(True)
    return nbr.cpu().numpy(), dist.cpu().numpy()


@pytest.mark.parametrize("n,d,k", [
    (65, 5, 1), (64, 4, 24), (129, 4, 24), (200, 31, 25), (321, 32, 56), (500, 33, 57),
    (1000, 3, 120), (4097, 6, 24), (2050, 260, 9), (777, 516, 5), (2, 7, 1), (25, 8, 24),
])
def test_plain_tiles(orc, ctx, n, d, k):
    rng = np.random.default_rng(n + d)
    X = rng.standard_normal((n, d)).astype(np.float32)
    X[n // 2] = X[0]
    nbr, dist = _knn(ctx, torch.from_numpy(X).cuda(), k, "fp32", False)
    rn, rd = orc.knn(X, k)
    assert np.array_equal(nbr, rn) and np.array_equal(dist, rd)


@pytest.mark.parametrize("name,make,k", [
    ("blobs", lambda: workloads.blobs(16001, 100, 12, (0.5, 2.0), 41), 16),
    ("k24", lambda: workloads.blobs(20000, 128, 40, (0.5, 1.0), 42), 24),
    ("k60", lambda: workloads.blobs(18000, 64, 9, (1.0, 1.0), 43), 60),
    ("overlap", lambda: workloads.blobs(15000, 96, 100, (1.0, 1.0), 44, box=1.0), 25),
    ("moons", lambda: workloads.get("moons_50k").points(20000), 7),
    ("duplicates", lambda: workloads.with_duplicates(
        workloads.blobs(25000, 32, 30, (0.5, 1.0), 45), 3000, 46), 9),
])
def test_pruned_tiles(ctx, name, make, k):
    X = torch.from_numpy(make()).cuda()
    assert X.shape[0] ** 2 * (X.shape[1] + 18) >= 2.5e10   # large enough to be pruned
    pn, pd = _knn(ctx, X, k, "fp32", True)
    un, ud = _knn(ctx, X, k, "fp32", False)
    assert np.array_equal(pn, un) and np.array_equal(pd, ud)


# uncertified rows: a few (each redone over its own list) or many (the FP32
# tiles over all lists)
@pytest.mark.parametrize("make,prec,k,few", [
    (lambda: workloads.get("blobs_100k").points(), "bf16x3", 16, True),
    (lambda: workloads.blobs(30000, 128, 15, (0.4, 2.0), 47), "bf16x3", 16, True),
    (lambda: workloads.blobs(30000, 128, 15, (0.4, 2.0), 47), "bf16x3", 20, False),
    (lambda: workloads.blobs(30000, 128, 15, (0.4, 2.0), 47), "bf16", 16, False),
], ids=["few", "few16", "many20", "bf16"])
def test_uncertified_rows_on_the_lists(ctx, make, prec, k, few):
    X = torch.from_numpy(make()).cuda()
    _, info = ctx.build(X, k, 2, 1, prec)
    assert 0 < info.uncertified_rows
    assert (info.uncertified_rows <= X.shape[0] // 32) == few
    pn, pd = _knn(ctx, X, k, prec, True)
    un, ud = _knn(ctx, X, k, "fp32", False)
    assert np.array_equal(pn, un) and np.array_equal(pd, ud)
