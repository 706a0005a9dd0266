"""The tensor tiles' candidate lists: rows at the edges of the query and key
tiles, k at the edges of the per-thread list lengths, masses of equal scores
that overflow a row's log, far keys before near ones, key lists split into
parts, and the masked pass with few foreign keys. Every row is exact whatever
the lists hold, so everything is compared bit for bit with the FP32 tiles."""
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


def _same(ctx, X, k, precs, prune=False):
    X = torch.from_numpy(np.ascontiguousarray(X, dtype=np.float32)).cuda()
    ctx.set_knn_pruning(False)
    rn, rd = ctx.knn_graph(X, k, "fp32")
    ctx.set_knn_pruning(prune)
    for prec in precs:
        nbr, dist = ctx.knn_graph(X, k, prec)
        assert torch.equal(nbr, rn) and torch.equal(dist, rd), prec
    ctx.set_knn_pruning(True)


ALL = ("bf16x3", "bf16", "fp8")


@pytest.mark.parametrize("n,d,k", [
    (64, 8, 1), (127, 64, 2), (128, 65, 3), (129, 32, 7), (150, 4, 8), (200, 128, 21),
    (255, 60, 22), (256, 16, 37), (257, 100, 38), (300, 129, 63), (513, 260, 21), (1000, 48, 63),
])
def test_edges(ctx, n, d, k):
    rng = np.random.default_rng(1000 * n + d)
    _same(ctx, rng.standard_normal((n, d)), k, ALL)


@pytest.mark.parametrize("k", [5, 16, 32, 50])
def test_equal_scores(ctx, k):
    # 700 copies of one point (every score equal), two-valued points, a grid
    rng = np.random.default_rng(k)
    X = rng.integers(0, 2, (2000, 6)).astype(np.float32)
    X[:700] = X[0]
    _same(ctx, X, k, ALL)
    _same(ctx, workloads.integer_grid(11, d=3), k, ("bf16x3",))


@pytest.mark.parametrize("k", [4, 16, 33])
def test_far_keys_first(ctx, k):
    # distances fall along the index, so every tile improves every row's list
    n = 3000
    X = np.zeros((n, 33), np.float32)
    X[:, 0] = np.geomspace(1e3, 1e-2, n)
    X[:, 1:] = np.random.default_rng(k).standard_normal((n, 32)).astype(np.float32) * 1e-3
    _same(ctx, X, k, ("bf16x3", "bf16"))


@pytest.mark.parametrize("k", [8, 21, 32, 45])
def test_split_lists(ctx, k):
    # overlapping clusters: most tiles list most keys, so the lists are split
    X = workloads.blobs(30000, 64, 150, (1.0, 1.0), 51, box=1.0)
    _same(ctx, X, k, ("bf16x3",), prune=True)


@pytest.mark.parametrize("n,far", [(129, 1), (257, 2), (600, 3), (1500, 40)])
def test_few_foreign_keys(orc, ctx, n, far):
    # one cluster and a few distant points: masked rows with few keys left
    rng = np.random.default_rng(n)
    X = rng.standard_normal((n, 20)).astype(np.float32)
    X[n - far:] += 50.0 * np.arange(1, far + 1, dtype=np.float32)[:, None]
    T, _ = ctx.emst_exact(torch.from_numpy(X).cuda(), "bf16x3")
    P = orc.prim_exact(X)
    ref, _ = ctx.emst_exact(torch.from_numpy(X).cuda(), "fp32")
    assert torch.equal(T.u, ref.u) and torch.equal(T.v, ref.v) and torch.equal(T.w, ref.w)
    assert T.W == pytest.approx(float(P.W), rel=1e-9)
