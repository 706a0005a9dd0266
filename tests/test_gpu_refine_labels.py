"""famst_refine on labels of the caller's own: closed under the kNN edges
(Algorithm 2's, or unions of its components: the grouped scans) and open ones
(kNN edges between components: the per-edge scans that test each candidate's
label), with the sweep cap at its ends. Against the oracle, bit for bit."""
import numpy as np
import pytest

import workloads

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


@pytest.fixture(scope="module")
def ctx(fam):
    return fam.Context(0)


def _case(orc, ctx, d, kind):
    X = workloads.blobs(3001, d, 12, (0.5, 1.5), 70 + d)
    Xd = torch.from_numpy(X).cuda()
    nbr, _ = ctx.knn_graph(Xd, 9)
    nb = nbr.cpu().numpy()
    G = orc.build_graph(nb)
    comp = orc.components(G).comp.copy()
    rng = np.random.default_rng(d)
    if kind == "unions":      # pairs of components under one label
        lab = comp // 2
    elif kind == "open":      # labels that cut through the kNN graph
        lab = rng.integers(0, 5, X.shape[0])
    else:
        lab = comp
    first = {}
    for l in lab.tolist():
        first.setdefault(int(l), len(first))
    comp = np.array([first[int(l)] for l in lab], np.int32)
    t = len(first)
    off = np.zeros(t + 1, np.int64)
    off[1:] = np.bincount(comp, minlength=t).cumsum()
    C = orc.Components(comp, np.argsort(comp, kind="stable").astype(np.int32), off)
    E = ctx.connect(Xd, torch.from_numpy(comp).cuda(), t, 4, 9)
    R = orc.random_edges(X, C, 4, 9)
    assert np.array_equal(E.u.cpu().numpy(), R.u) and np.array_equal(E.v.cpu().numpy(), R.v)
    return X, Xd, nbr, G, C, E, R


@pytest.mark.parametrize("d", [16, 32, 64, 100, 128, 200])
@pytest.mark.parametrize("kind", ["components", "unions", "open"])
def test_refine(orc, ctx, d, kind):
    X, Xd, nbr, G, C, E, R = _case(orc, ctx, d, kind)
    sweeps, delta = ctx.refine(Xd, nbr, torch.from_numpy(C.comp).cuda(), E)
    deltas, _ = orc.refine(X, G, C, R)   # in place
    assert delta == [int(x) for x in deltas] and sweeps == len(deltas)
    for a, b in ((E.u, R.u), (E.v, R.v), (E.w, R.w)):
        assert np.array_equal(a.cpu().numpy(), b)


@pytest.mark.parametrize("kind", ["components", "open"])
def test_sweep_cap(orc, fam, ctx, kind):
    X, Xd, nbr, G, C, E, R = _case(orc, ctx, 64, kind)
    comp = torch.from_numpy(C.comp).cuda()
    need = len(orc.refine(X, G, C, R)[0])
    assert need > 2
    for cap in (1, 2, need - 1):
        with pytest.raises(fam.FamstError) as e:
            ctx.refine(Xd, nbr, comp, E.clone(), max_iters=cap)
        assert e.value.name == "FAMST_ERR_NO_CONVERGENCE"
    sweeps, _ = ctx.refine(Xd, nbr, comp, E.clone(), max_iters=need)
    assert sweeps == need
