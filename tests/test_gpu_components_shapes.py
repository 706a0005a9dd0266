"""Component labels on graphs that stress the rounds before the final hooks:
paths in ascending, descending and random id order, a hub every vertex points
at, many tiny components, one neighbour per vertex. Against the oracle."""
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


def _graph(kind, n, rng):
    i = np.arange(n)
    if kind == "path":
        return np.stack([np.where(i < n - 1, i + 1, n - 2), np.where(i > 0, i - 1, 1)], 1)
    if kind == "hub_high":
        return np.where(i == n - 1, 0, n - 1)[:, None]
    if kind == "hub_low":
        return np.where(i == 0, n - 1, 0)[:, None]
    if kind == "pairs":
        return (i ^ 1)[:, None]
    if kind == "random":   # sparse: several components
        return (i[:, None] + 1 + rng.integers(0, n - 1, (n, 1))) % n
    g = rng.integers(0, 40, n)   # dense inside 40 groups
    order = np.argsort(g, kind="stable")
    out = np.empty((n, 16), np.int64)
    for c in range(40):
        m = order[g[order] == c]
        r = rng.integers(1, len(m), (len(m), 16))
        out[m] = m[(np.arange(len(m))[:, None] + r) % len(m)]
    return out


@pytest.mark.parametrize("kind,n", [("path", 3000), ("path", 100001), ("hub_high", 5000),
                                    ("hub_low", 5000), ("pairs", 10000), ("random", 20000),
                                    ("groups", 30000)])
@pytest.mark.parametrize("shuffle", [False, True])
def test_components(orc, ctx, kind, n, shuffle):
    rng = np.random.default_rng(n)
    nbr = _graph(kind, n, rng)
    if shuffle:
        p = rng.permutation(n)
        q = np.empty_like(nbr)
        q[p] = p[nbr]
        nbr = q
    nbr = np.ascontiguousarray(nbr, dtype=np.int32)
    assert np.all(nbr != np.arange(n)[:, None]) and nbr.min() >= 0 and nbr.max() < n
    comp, t = ctx.components(torch.from_numpy(nbr).cuda())
    C = orc.components(orc.build_graph(nbr))
    assert t == C.t
    assert np.array_equal(comp.cpu().numpy(), C.comp)
