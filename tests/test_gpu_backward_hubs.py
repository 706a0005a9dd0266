"""The gradient of trees with many vertices of middling degree: ordering each
vertex's edges by ranks costs the sum of the squared degrees, so such trees are
radix sorted although no single degree is large. Both ways against the FP64
oracle; the way is seen in the number of launches."""
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


def hubs(n, leaves, rng):
    """A chain of hubs with `leaves` leaves each (0: a path), ids and edges shuffled."""
    i = np.arange(n)
    h = i // (leaves + 1) * (leaves + 1)
    par = np.where(i == h, np.maximum(h - (leaves + 1), 0), h)
    p, o = rng.permutation(n), rng.permutation(n - 1)
    return p[i[1:]][o].astype(np.int32), p[par[1:]][o].astype(np.int32)


# sums of squared degrees on either side of 4e7 + 70 m, one degree beyond 2048
@pytest.mark.parametrize("n,leaves,sorted_", [(30001, 1800, True), (30000, 200, False),
                                              (9001, 2040, False), (400, 398, False),
                                              (5000, 3000, True), (2, 0, False)])
@pytest.mark.parametrize("d", [3, 40])
def test_hubs(orc, ctx, n, leaves, sorted_, d):
    rng = np.random.default_rng(n + d)
    X = rng.standard_normal((n, d)).astype(np.float32)
    tu, tv = hubs(n, leaves, rng)
    Xd = torch.from_numpy(X).cuda()

    def run(u, v):
        before = ctx.launches
        g = ctx.mst_backward(Xd, torch.from_numpy(u).cuda(), torch.from_numpy(v).cuda(), 1.0)
        return g.cpu().numpy(), ctx.launches - before
    g, launches = run(tu, tv)
    _, path = run(*hubs(n, 0, rng))
    assert (launches > path + 3) == sorted_
    g64 = orc.mst_grad(X, tu, tv)
    deg = np.bincount(np.concatenate([tu, tv]), minlength=n)[:, None].astype(np.float64)
    assert np.all(np.abs(g - g64) <= deg * (d + 4 + deg) * 2.0 ** -24 + 1e-7)
