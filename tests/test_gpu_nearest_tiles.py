"""The nearest-pair connect at the sizes of its tensor-core pass: components
that end inside a tile or span several, many components per 16 columns,
lambda at its ends, every operand width, points of one component only in the
last tile, and inputs whose ties overflow the survivor buffer. Against the
oracle, bit for bit."""
import numpy as np
import pytest

import workloads

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


@pytest.mark.parametrize("n,d,t,lam,even", [
    (4096, 64, 2, 1, True), (4097, 65, 3, 32, True), (5003, 128, 16, 5, False),
    (6000, 130, 300, 3, False), (4352, 256, 7, 10, True), (4500, 3, 40, 8, False),
    (20011, 32, 11, 5, False), (4100, 16, 1000, 2, True),
])
def test_tiles(orc, ctx, n, d, t, lam, even):
    rng = np.random.default_rng(n + d)
    X = (rng.standard_normal((n, d)) + 4.0 * rng.standard_normal((t, d))[np.arange(n) % t])
    X = np.ascontiguousarray(X, dtype=np.float32)
    lab = np.arange(n) % t
    if not even:   # sizes from one point to a large share
        lab = np.minimum((rng.random(n) ** 3 * t).astype(np.int64), t - 1)
        lab[:t] = np.arange(t)
    X[n - 1] = X[0]   # a pair at distance zero when the two differ in component
    _check(orc, ctx, X, lab, lam)


def test_ties_overflow_the_survivors(orc, ctx):
    # 2500 points at one distance from 2000 nearly coincident ones: five
    # million cross pairs within the rounding bounds of the smallest
    rng = np.random.default_rng(4)
    a = rng.standard_normal((2500, 64))
    a[:, 0] = 0.0
    a /= np.linalg.norm(a, axis=1, keepdims=True)
    b = 1e-5 * rng.standard_normal((2000, 64))
    b[:, 0] += 30.0
    X = np.ascontiguousarray(np.concatenate([a, b]), dtype=np.float32)
    _check(orc, ctx, X, (np.arange(4500) >= 2500).astype(np.int64), 7)
