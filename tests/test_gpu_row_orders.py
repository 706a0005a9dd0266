"""Clouds whose row index has a period (pixel grids, interleaved labels): the
lists equal the FP32 tiles', and no more rows of the tensor passes lose their
certificate than of the same points in random order (within 1 %)."""
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


def grid(w, n, d=3):
    rng = np.random.default_rng(w)
    X = np.zeros((n, d))
    X[:, 0], X[:, 1] = np.arange(n) % w, np.arange(n) // w
    return np.ascontiguousarray(X + rng.uniform(-0.2, 0.2, X.shape), dtype=np.float32)


def labels(p, n, d):
    rng = np.random.default_rng(p)
    c = rng.standard_normal((p, d)) * 20
    return np.ascontiguousarray(c[np.arange(n) % p] + rng.standard_normal((n, d)), dtype=np.float32)


CLOUDS = [grid(64, 3968), grid(32, 4001), grid(64, 9000, 5), labels(32, 8000, 5),
          labels(64, 3999, 33)]


@pytest.mark.parametrize("c", range(len(CLOUDS)))
@pytest.mark.parametrize("k", [1, 10, 32])
def test_knn(ctx, c, k):
    X = torch.from_numpy(CLOUDS[c]).cuda()
    rn, rd = ctx.knn_graph(X, k, "fp32")
    for prec in ("bf16x3", "bf16", "fp8"):
        nbr, dist = ctx.knn_graph(X, k, prec)
        assert torch.equal(nbr, rn) and torch.equal(dist, rd), prec
    _, info = ctx.build(X, k, 2, 1, "bf16x3")
    order = torch.from_numpy(np.random.default_rng(0).permutation(len(X))).cuda()
    _, mixed = ctx.build(X[order].contiguous(), k, 2, 1, "bf16x3")
    assert info.uncertified_rows <= mixed.uncertified_rows + len(X) // 100


@pytest.mark.parametrize("c", [0, 3])
def test_emst(ctx, c):
    X = torch.from_numpy(CLOUDS[c]).cuda()
    T, _ = ctx.emst_exact(X, "bf16x3")
    ref, _ = ctx.emst_exact(X, "fp32")
    assert torch.equal(T.u, ref.u) and torch.equal(T.v, ref.v) and torch.equal(T.w, ref.w)


def test_batch(ctx):
    # offsets along (1, 1, 0) and (0, 1, 1) in 64ths: the +-1 projection that
    # orders a batch's rows is exactly the same along every diagonal of the grid
    rng = np.random.default_rng(5)
    clouds = []
    for w, n in ((32, 3200), (128, 8064)):
        a, b = rng.integers(-12, 13, (2, n)) / 64.0
        i = np.arange(n)
        clouds.append(np.stack([i % w + a, i // w + a + b, b], 1).astype(np.float32))
    clouds.append(labels(32, 1500, 16))
    flat = torch.from_numpy(np.concatenate([c.ravel() for c in clouds])).cuda()
    off = np.cumsum([0] + [len(c) for c in clouds]).astype(np.int64)
    dims = np.array([c.shape[1] for c in clouds], np.int32)
    trees, W, t, info = ctx.build_batched(flat, off, dims, 16, 3, 5, "bf16x3")
    assert info.tensor_clouds >= 2   # the two grids (the small cloud may take the FP32 tiles)
    mixed = np.concatenate([rng.permutation(c).ravel() for c in clouds])
    _, _, _, info2 = ctx.build_batched(torch.from_numpy(mixed).cuda(), off, dims, 16, 3, 5, "bf16x3")
    assert info.uncertified_rows <= info2.uncertified_rows + off[-1] // 100
    for b, c in enumerate(clouds):
        one, _ = ctx.build(torch.from_numpy(c).cuda(), 16, 3, 5 + b, "fp32")
        assert torch.equal(trees[b].w, one.w) and t[b] > 0
