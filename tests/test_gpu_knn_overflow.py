"""kNN graphs of finite points whose squared norms leave the FP32 range: scores
of the tensor tiles are then infinite or no numbers, and no row may be certified
by them. The oracle's lists, whatever the precision asked for."""
import numpy as np
import pytest

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


def camps(n, d, seed):
    """Clusters 1e16 apart around three far places: two whose squared norms
    overflow, and one near the origin whose norms are ordinary."""
    rng = np.random.default_rng(seed)
    c = rng.standard_normal((n // 40 + 1, d)) * 1e16
    c[:, 0] += np.array([-3e19, 3e19, 0.0])[np.arange(len(c)) % 3]
    X = c[np.arange(n) % len(c)] + rng.standard_normal((n, d)) * 1e14
    return np.ascontiguousarray(X, dtype=np.float32)


# below the size that prunes tiles
@pytest.mark.parametrize("n,d,k", [(1500, 8, 6), (1001, 31, 40)])
@pytest.mark.parametrize("prec", ["bf16x3", "bf16", "fp8"])
def test_lists(orc, ctx, n, d, k, prec):
    X = camps(n, d, n + d)
    nbr, dist = ctx.knn_graph(torch.from_numpy(X).cuda(), k, prec)
    rn, rd = orc.knn(X, k)
    np.testing.assert_array_equal(nbr.cpu().numpy(), rn)
    np.testing.assert_array_equal(dist.cpu().numpy(), rd)


def test_batch(orc, ctx):
    # a chain of far places, so that the trees have finite edges only
    X = camps(700, 16, 1) * np.float32(0.1)
    X[:, 0] += (np.arange(700) % 4).astype(np.float32) * np.float32(1.5e19)
    Xs = [X, np.random.default_rng(2).standard_normal((900, 16)).astype(np.float32)]
    flat = torch.from_numpy(np.concatenate([x.reshape(-1) for x in Xs])).cuda()
    trees, W, t, _ = ctx.build_batched(flat, np.array([0, 700, 1600], np.int64),
                                       np.array([16, 16], np.int32), 6, 3, 5, "bf16x3")
    for b, x in enumerate(Xs):
        ref = orc.famst(x, 6, 3, 5)
        assert int(t[b]) == ref.C.t
        np.testing.assert_array_equal(np.sort(trees[b].w.cpu().numpy()), np.sort(ref.tree.w))


def spread(n, d, seed):
    """One cloud whose squared distances lie around the end of the FP32 range:
    many pairs overflow, but no point's nearest ones."""
    rng = np.random.default_rng(seed)
    return np.ascontiguousarray(rng.standard_normal((n, d)) * 3.5e18, dtype=np.float32)


# sizes whose tiles are pruned where the norms allow it
@pytest.mark.parametrize("n,d,k,precs", [(5000, 12, 8, ("bf16x3", "bf16", "fp32")),
                                         (28000, 16, 10, ("fp32", "bf16x3"))])
@pytest.mark.parametrize("cloud", [camps, spread])
def test_pruned_sizes(orc, ctx, n, d, k, precs, cloud):
    X = cloud(n, d, n)
    rows = np.random.default_rng(1).choice(n, 1500, replace=False).astype(np.int32)
    rn, rd = orc.knn_rows(X, k, rows)
    for prec in precs:
        nbr, dist = ctx.knn_graph(torch.from_numpy(X).cuda(), k, prec)
        np.testing.assert_array_equal(nbr.cpu().numpy()[rows], rn)
        np.testing.assert_array_equal(dist.cpu().numpy()[rows], rd)
