"""Boruvka's minimum passes: graphs whose warps hold one, two and many
components, with masses of equal weights, at sizes around the edges taken per
lane. The tree must be Kruskal's edge for edge (ties by the smaller, then the
larger end)."""
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


def _keys(w, u, v):
    w, u, v = (np.asarray(x) for x in (w, u, v))
    a, b = np.minimum(u, v), np.maximum(u, v)
    o = np.lexsort((b, a, w))
    return np.stack([w[o].view(np.int32).astype(np.int64), a[o], b[o]], 1)


@pytest.mark.parametrize("n,k,levels", [
    (2, 1, 1), (33, 1, 2), (127, 3, 1), (128, 8, 3), (1000, 16, 4), (1001, 31, 2),
    (4099, 33, 1000), (20000, 7, 1), (20000, 16, 50),
])
def test_tree(orc, ctx, n, k, levels):
    rng = np.random.default_rng(n + k)
    step = rng.integers(1, n, (n, k))
    step[:, 0] = 1   # a ring: connected
    nbr = ((np.arange(n)[:, None] + step) % n).astype(np.int32)
    a, b = np.minimum(np.arange(n)[:, None], nbr), np.maximum(np.arange(n)[:, None], nbr)
    dist = ((a * 7919 + b * 104729) % levels).astype(np.float32) + 0.5   # one weight per edge
    # rows sorted by (distance, id), as a kNN graph's are
    o = np.lexsort((nbr, dist), axis=1)
    nbr, dist = np.take_along_axis(nbr, o, 1), np.take_along_axis(dist, o, 1)
    tu, tv, tw, W = ctx.mst(n, torch.from_numpy(nbr).cuda(), torch.from_numpy(dist).cuda(), None)
    ref = orc.kruskal(n, nbr, dist, None)
    assert np.array_equal(_keys(tw.cpu(), tu.cpu(), tv.cpu()), _keys(ref.w, ref.u, ref.v))
