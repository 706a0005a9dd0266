"""NN-Descent's local joins: row widths and sample sizes on both sides of the
rule between one warp and one block per vertex, tiles of few and of many new
candidates, remainders of the partials' order. Lists, updates and pair counts
equal the oracle's."""
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


@pytest.mark.parametrize("n,d,k,S", [
    (40, 4, 3, 1), (300, 12, 5, 2), (700, 28, 9, 4), (900, 32, 16, 16), (901, 36, 17, 17),
    (1500, 128, 16, 16), (800, 148, 16, 16), (800, 172, 16, 16), (800, 176, 16, 16),
    (600, 64, 31, 32), (600, 60, 32, 32), (500, 300, 8, 4), (500, 130, 8, 6),
])
def test_join(orc, ctx, n, d, k, S):
    X = workloads.blobs(n, d, 5, (0.5, 1.5), n + d)
    nbr, dist, it, upd, prs = ctx.knn_nndescent(torch.from_numpy(np.ascontiguousarray(X)).cuda(),
                                                k, S, 8, 0.0, 3)
    r = orc.nndescent(X, k, S, 8, 0.0, 3)
    assert it == r.iters and upd.tolist() == r.updates.tolist() and prs.tolist() == r.pairs.tolist()
    assert np.array_equal(nbr.cpu().numpy(), r.nbr) and np.array_equal(dist.cpu().numpy(), r.dist)
