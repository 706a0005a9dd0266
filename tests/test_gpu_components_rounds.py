"""Component labels where the lowering rounds' slices of a neighbour list start
beyond it, overlap or end with it, on graphs whose rounds leave long chains.
Against the oracle."""
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


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 11, 17])
@pytest.mark.parametrize("order", ["ascending", "descending", "random"])
def test_strips(orc, ctx, k, order):
    # strips of 700 vertices, each joined to k of the 2 k nearest in its strip
    rng = np.random.default_rng(k)
    n, s = 9100, 700
    i = np.arange(n)[:, None]
    step = np.concatenate([np.arange(-k, 0), np.arange(1, k + 1)])
    pick = np.argsort(rng.random((n, 2 * k)), axis=1)[:, :k]
    nbr = i // s * s + (i % s + step[pick]) % s
    p = {"ascending": np.arange(n), "descending": np.arange(n)[::-1],
         "random": rng.permutation(n)}[order]
    q = np.empty_like(nbr)
    q[p] = p[nbr]
    q = np.ascontiguousarray(q, dtype=np.int32)
    comp, t = ctx.components(torch.from_numpy(q).cuda())
    C = orc.components(orc.build_graph(q))
    assert t == C.t
    assert np.array_equal(comp.cpu().numpy(), C.comp)
