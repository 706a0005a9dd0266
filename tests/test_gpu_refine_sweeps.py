"""famst_refine with more edges than go to the per-edge kernel from the first
sweep (65,536) and enough work for the grouped route: the sweep-synchronous
scans at three operand widths, with the sweep cap at its ends. Against the
oracle, bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - deselected on CPU runs
    pytest.skip("needs a CUDA device", allow_module_level=True)


@pytest.fixture(scope="module")
def fam():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2507_14261_gb300 as P
    return P


@pytest.mark.parametrize("d,k,lam", [(64, 30, 16), (128, 30, 9), (200, 20, 8)])
def test_sweeps(orc, fam, d, k, lam):
    ctx = fam.Context(0)
    rng = np.random.default_rng(d)
    c = rng.uniform(-10, 10, (130, d))
    n = 130 * 40
    X = np.ascontiguousarray((c[np.arange(n) % 130] + 0.3 * rng.standard_normal((n, d)))
                             [rng.permutation(n)], dtype=np.float32)
    Xd = torch.from_numpy(X).cuda()
    nbr, _ = ctx.knn_graph(Xd, k)
    comp, t = ctx.components(nbr)
    E = ctx.connect(Xd, comp, t, lam, 3)
    m = E.u.numel()
    assert t == 130 and m > 65536 and m * k * d >= 2.3e8 + 92.0 * n * k
    G = orc.build_graph(nbr.cpu().numpy())
    C = orc.components(G)
    R = orc.random_edges(X, C, lam, 3)
    deltas, _ = orc.refine(X, G, C, R)   # in place
    need = len(deltas)
    assert need > 2
    for cap in (1, 2, need - 1):
        with pytest.raises(fam.FamstError) as e:
            ctx.refine(Xd, nbr, comp, E.clone(), max_iters=cap)
        assert e.value.name == "FAMST_ERR_NO_CONVERGENCE"
    F = E.clone()
    assert ctx.refine(Xd, nbr, comp, F, max_iters=need)[0] == need
    sweeps, delta = ctx.refine(Xd, nbr, comp, E)
    assert delta == [int(x) for x in deltas] and sweeps == need
    for a, b, f in ((E.u, R.u, F.u), (E.v, R.v, F.v), (E.w, R.w, F.w)):
        assert np.array_equal(a.cpu().numpy(), b) and torch.equal(a, f)
