"""Alg. 3 of a build on the BF16 rows, at the edges of its layouts: row
widths of one to four 64-column blocks, lambda^2 draws in one, two and four
registers, two to several hundred components (pair enumeration). The build's
tree must be the oracle's edge for edge."""
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


def _groups(groups, per, d, seed):
    rng = np.random.default_rng(seed)
    c = rng.standard_normal((groups, d)).astype(np.float32) * 40.0
    X = np.repeat(c, per, axis=0) + rng.standard_normal((groups * per, d)).astype(np.float32)
    return np.ascontiguousarray(X, dtype=np.float32)


@pytest.mark.parametrize("groups,per,d,lam", [
    (2, 40, 64, 1), (3, 30, 32, 5), (17, 20, 100, 6), (40, 25, 128, 8),
    (300, 9, 128, 10), (12, 30, 192, 9), (25, 20, 256, 11), (500, 8, 64, 3),
])
def test_build(orc, ctx, groups, per, d, lam):
    X = _groups(groups, per, d, groups + d)
    tree, info = ctx.build(torch.from_numpy(X).cuda(), 5, lam, 7, "fp32")
    ref = orc.famst(X, 5, lam, 7)
    assert info.t >= groups
    assert tree.W == pytest.approx(ref.tree.W, rel=1e-12)

    def keys(w, u, v):
        w, u, v = (np.asarray(x) for x in (w, u, v))
        a, b = np.minimum(u, v), np.maximum(u, v)
        o = np.lexsort((b, a, w))
        return np.stack([w[o].view(np.int32).astype(np.int64), a[o], b[o]], 1)

    assert np.array_equal(keys(tree.w.cpu(), tree.u.cpu(), tree.v.cpu()),
                          keys(ref.tree.w, ref.tree.u, ref.tree.v))
