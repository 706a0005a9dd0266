"""The nearest-pair connect with so many component pairs that its first launch
only lowers the bounds and the search follows over all rows. Against the oracle,
bit for bit."""
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


def _check(orc, ctx, X, labels, lam):
    """Components given by labels (numbered by their smallest member)."""
    first = {}
    for l in labels.tolist():
        first.setdefault(l, len(first))
    comp = np.array([first[l] for l in labels.tolist()], np.int32)
    t = len(first)
    off = np.zeros(t + 1, np.int64)
    off[1:] = np.bincount(comp, minlength=t).cumsum()
    members = np.argsort(comp, kind="stable").astype(np.int32)
    C = orc.Components(comp, members, off)
    E = ctx.connect_nearest(torch.from_numpy(X).cuda(), torch.from_numpy(comp).cuda(), t, lam)
    R = orc.nearest_edges(X, C, lam)
    for a, b in ((E.u, R.u), (E.v, R.v), (E.w, R.w), (E.ci, R.ci), (E.cj, R.cj)):
        assert np.array_equal(a.cpu().numpy(), b)


@pytest.mark.parametrize("n,d,t,lam", [(20000, 32, 300, 32), (20011, 64, 600, 2)])
def test_bounds_before_the_search(orc, ctx, n, d, t, lam):
    # room for a search only after a launch that lowers the bounds
    rng = np.random.default_rng(n)
    X = rng.standard_normal((n, d)) + 6.0 * rng.standard_normal((t, d))[np.arange(n) % t]
    _check(orc, ctx, np.ascontiguousarray(X, dtype=np.float32), np.arange(n) % t, lam)
