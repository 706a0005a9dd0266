"""Nearest-pair connect of finite points whose squared norms leave the FP32
range, or come close: the tiles' thresholds are squares and decide nothing
there, so the edges have to come from canonical distances all the same."""
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


# half the distance of two camps of clusters: all squared norms overflow (3e19),
# some distances do (0.9223e19), the norms alone are in range (1e18, 1e17)
@pytest.mark.parametrize("half", [3e19, 0.9223e19, 1e18, 1e17])
@pytest.mark.parametrize("d", [16, 128])
def test_overflow(orc, ctx, d, half):
    rng = np.random.default_rng(d)
    comps, per = 40, 30   # 1200 points: the tiles' side of the rule
    c = rng.standard_normal((comps, d)) * 1e16
    c[:, 0] += np.where(np.arange(comps) % 2, half, -half)
    X = np.repeat(c, per, axis=0) + rng.standard_normal((comps * per, d)) * 1e14
    X = np.ascontiguousarray(X[rng.permutation(len(X))], dtype=np.float32)
    Xd = torch.from_numpy(X).cuda()
    nbr, _ = ctx.knn_graph(Xd, 5, "fp32")
    C = orc.components(orc.build_graph(nbr.cpu().numpy()))
    assert C.t == comps
    R = orc.nearest_edges(X, C, 7)
    E = ctx.connect_nearest(Xd, torch.from_numpy(C.comp).cuda(), C.t, 7)
    for a, b in ((E.u, R.u), (E.v, R.v), (E.w, R.w), (E.ci, R.ci), (E.cj, R.cj)):
        assert np.array_equal(a.cpu().numpy(), b)
