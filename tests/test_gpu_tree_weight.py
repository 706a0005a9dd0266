"""famst_tree_weight with points that are not ordinary numbers. The call takes
any X: an edge that touches an infinity or a NaN has to show in W64, and zeros
of either sign, subnormals and the largest floats have their exact FP64 value."""
import math

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


BIG = float(np.finfo(np.float32).max)
VALUES = [math.inf, -math.inf, math.nan, BIG, -BIG, 0.0, -0.0, 1e-45, -1.1e-38, 1.17549435e-38]


@pytest.mark.parametrize("d", [8, 7])   # 16-byte rows and the others
@pytest.mark.parametrize("value", VALUES)
def test_tree_weight_values(ctx, d, value):
    n = 300
    X = np.random.default_rng(d).standard_normal((n, d)).astype(np.float32)
    X[17, 3] = np.float32(value)
    X[18, 3] = np.float32(value)   # next to it: inf - inf, or a difference of zero
    tu = torch.arange(n - 1, dtype=torch.int32, device="cuda")
    tw = torch.ones(n - 1, device="cuda")
    W, W64 = ctx.tree_weight(torch.from_numpy(X).cuda(), tu, tu + 1, tw)
    with np.errstate(invalid="ignore"):
        ref = float(np.sqrt((np.diff(X.astype(np.float64), axis=0) ** 2).sum(1)).sum())
    assert W == n - 1
    if math.isnan(ref):
        assert math.isnan(W64)
    else:   # n sums of d products, each rounded once in FP64
        assert W64 == pytest.approx(ref, rel=(n + d) * 2.0 ** -52)
