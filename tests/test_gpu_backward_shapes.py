"""The gradient of the tree weight on every lane layout of its kernels and
both ways of ordering a vertex's edges: widths at the edges of the layouts,
vertices beyond the rank limit (a star: the radix sort), duplicates (edges of
length zero), bad ids and non-finite points. Checked against the FP64 oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - deselected on CPU runs
    pytest.skip("needs a CUDA device", allow_module_level=True)


@pytest.fixture(scope="module")
def fam():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2507_14261_gb300 as P
    return P


@pytest.fixture(scope="module")
def ctx(fam):
    return fam.Context(0)


def _tree(kind, n, rng):
    """Edges of a spanning tree in random order and orientation."""
    v = np.arange(1, n)
    if kind == "star":
        u = np.zeros(n - 1, np.int64)
    elif kind == "path":
        u = v - 1
    else:   # random attachment, a few hubs
        u = (rng.random(n - 1) ** 3 * v).astype(np.int64)
    p = rng.permutation(n)
    u, v = p[u], p[v]
    flip = rng.random(n - 1) < 0.5
    u, v = np.where(flip, v, u), np.where(flip, u, v)
    o = rng.permutation(n - 1)
    return u[o].astype(np.int32), v[o].astype(np.int32)


@pytest.mark.parametrize("d", [1, 2, 3, 4, 5, 8, 9, 16, 17, 32, 33, 64, 65, 128, 129, 200, 256, 257, 520])
@pytest.mark.parametrize("kind,n", [("random", 1003), ("star", 2050), ("path", 9), ("random", 2)])
def test_gradient(orc, ctx, kind, n, d):
    rng = np.random.default_rng(1000 * d + n)
    X = rng.standard_normal((n, d)).astype(np.float32)
    if n > 100:
        X[50:60] = X[40:50]
    tu, tv = _tree(kind, n, rng)
    if n > 100:   # some edges of length zero
        tu[:3], tv[:3] = np.arange(50, 53), np.arange(40, 43)
    g = ctx.mst_backward(torch.from_numpy(X).cuda(), torch.from_numpy(tu).cuda(),
                         torch.from_numpy(tv).cuda(), 2.0).cpu().numpy()
    g64 = 2.0 * orc.mst_grad(X, tu, tv)
    # FP32 terms of magnitude <= 1 with relative error (d + 4) 2^-24, and one
    # rounding of a sum of at most deg per addition
    deg = np.bincount(np.concatenate([tu, tv]), minlength=n)[:, None].astype(np.float64)
    assert np.all(np.abs(g - g64) <= 2.0 * deg * (d + 4 + deg) * 2.0 ** -24 + 1e-7)


@pytest.mark.parametrize("d", [3, 64])
def test_bad_inputs(fam, ctx, d):
    X = torch.randn((300, d), device="cuda")
    tu = torch.arange(1, 300, dtype=torch.int32, device="cuda")
    tv = tu - 1
    for bad in (-1, 300):
        t = tu.clone()
        t[17] = bad
        with pytest.raises(fam.FamstError) as e:
            ctx.mst_backward(X, t, tv)
        assert e.value.name == "FAMST_ERR_INVALID_ARG"
    Y = X.clone()
    Y[299, d - 1] = float("nan")
    with pytest.raises(fam.FamstError) as e:
        ctx.mst_backward(Y, tu, tv)
    assert e.value.name == "FAMST_ERR_NONFINITE"
    assert torch.isfinite(ctx.mst_backward(X, tu, tv)).all()
