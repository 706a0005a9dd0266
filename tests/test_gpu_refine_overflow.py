"""Alg. 4's grouped sweeps where squares leave the FP32 range: finite points far
apart, so that an edge's weight, its squared bound or a point's squared norm
overflows. The tensor-core filter may then rule nothing out, and every decision
falls on the canonical distances: edges and sweeps equal the oracle's."""
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


def two_camps(half, d, seed, per=8, comps=150):
    """`comps` clusters of `per` points, half of them around +half and half
    around -half in coordinate 0; clusters 1e16 apart, points 1e14."""
    rng = np.random.default_rng(seed)
    c = rng.standard_normal((comps, d)) * 1e16
    c[:, 0] = np.where(np.arange(comps) % 2, half, -half) + rng.uniform(-1e16, 1e16, comps)
    X = np.repeat(c, per, axis=0) + rng.standard_normal((comps * per, d)) * 1e14
    return np.ascontiguousarray(X[rng.permutation(len(X))], dtype=np.float32)


def _edges(u, v, w):
    a = np.stack([np.minimum(u, v), np.maximum(u, v), np.asarray(w).view(np.int32)]).astype(np.int64)
    return a[:, np.lexsort(a)]


# 0.921e19: weights of 1.842e19 are finite, but their square with the BF16 rows'
# errors is not; 3e19: weights between the camps and all squared norms overflow
@pytest.mark.parametrize("half", [0.921e19, 3e19])
@pytest.mark.parametrize("d,k,lam,per", [(32, 3, 6, 8), (100, 3, 6, 8), (256, 12, 7, 14)])
def test_overflow(orc, ctx, d, k, lam, per, half):
    X = two_camps(half, d, d, per)
    ref = orc.famst(X, k, lam, 11)
    assert len(ref.E) > 65536   # the sweeps are grouped; with d = 256 in famst_refine too
    Xd, comp = torch.from_numpy(X).cuda(), torch.from_numpy(ref.C.comp).cuda()
    nbr, _ = ctx.knn_graph(Xd, k, "fp32")
    assert np.array_equal(nbr.cpu().numpy(), ref.nbr)
    E = ctx.connect(Xd, comp, ref.C.t, lam, 11)
    sweeps, delta = ctx.refine(Xd, nbr, comp, E)
    assert delta == [int(x) for x in ref.deltas] and sweeps == len(ref.deltas)
    for a, b in ((E.u, ref.E.u), (E.v, ref.E.v), (E.w, ref.E.w)):
        assert np.array_equal(a.cpu().numpy(), b)
    tree, info = ctx.build(Xd, k, lam, 11, "fp32")
    assert info.t == ref.C.t and info.refine_sweeps == len(ref.deltas)
    assert info.first_delta == ref.deltas[0]
    assert np.array_equal(_edges(tree.u.cpu().numpy(), tree.v.cpu().numpy(), tree.w.cpu().numpy()),
                          _edges(ref.tree.u, ref.tree.v, ref.tree.w))
