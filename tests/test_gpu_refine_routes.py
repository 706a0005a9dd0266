"""Alg. 4 on both sides of its rules: per edge with few edges, grouped sweeps
with many, inside a build and through famst_refine. Edges equal the oracle's."""
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


# 200 groups: 19,900 pairs; lambda 3 / 4: 59,700 / 79,600 edges (65,536 between);
# d = 256, lambda 6: m k d = 2.8e8, grouped in famst_refine too
@pytest.mark.parametrize("d,k,lam", [(32, 6, 3), (32, 6, 4), (100, 5, 4), (256, 9, 6)])
def test_routes(orc, ctx, d, k, lam):
    rng = np.random.default_rng(d + lam)
    c = rng.standard_normal((200, d)).astype(np.float32) * 30.0
    X = np.repeat(c, 18, axis=0) + rng.standard_normal((3600, d)).astype(np.float32)
    X = np.ascontiguousarray(X[rng.permutation(3600)], dtype=np.float32)
    Xd = torch.from_numpy(X).cuda()
    ref = orc.famst(X, k, lam, 11)
    tree, info = ctx.build(Xd, k, lam, 11, "fp32")
    assert info.t == ref.C.t and info.refine_sweeps == len(ref.deltas)
    assert info.first_delta == ref.deltas[0]
    assert tree.W == pytest.approx(ref.tree.W, rel=1e-12)
    nbr, _ = ctx.knn_graph(Xd, k, "fp32")
    E = ctx.connect(Xd, torch.from_numpy(ref.C.comp).cuda(), ref.C.t, lam, 11)
    sweeps, delta = ctx.refine(Xd, nbr, torch.from_numpy(ref.C.comp).cuda(), E)
    assert delta == [int(x) for x in ref.deltas] and sweeps == len(ref.deltas)
    for a, b in ((E.u, ref.E.u), (E.v, ref.E.v), (E.w, ref.E.w)):
        assert np.array_equal(a.cpu().numpy(), b)
