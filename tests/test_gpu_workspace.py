"""Workspace of Phase 1: the tensor tiles' logs (1 MB per CTA that can be
resident) are counted for the work items a call can have, and not at all where
the FP32 tiles do the work. The same calls then run in what was counted."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - deselected on CPU runs
    pytest.skip("needs a CUDA device", allow_module_level=True)

MB = 1 << 20


@pytest.fixture(scope="module")
def fam():
    import __graft_entry__
    __graft_entry__.build()
    import paper_2507_14261_gb300 as P
    return P


def test_logs_by_items(fam):
    ctx = fam.Context(0)
    sms = torch.cuda.get_device_properties(0).multi_processor_count

    def query(n, prec):
        return ctx.workspace_query(n, 64, 16, 5, 50, prec)
    # 4096 points: 32 query tiles, lists too short to be split; 20,000: every SM.
    # Everything else grows with n.
    assert query(20000, "bf16x3") - query(4096, "bf16x3") >= (sms - 32) * MB
    assert query(30000, "bf16x3") - query(30000, "fp32") >= sms * MB
    ctx.set_knn_pruning(False)
    assert query(20000, "bf16x3") - query(4096, "bf16x3") >= (sms - 32) * MB


@pytest.mark.parametrize("n,prec", [(4096, "bf16x3"), (4097, "bf16x3"), (5000, "bf16x3"),
                                    (5000, "fp8"), (8300, "bf16"), (30000, "fp32")])
@pytest.mark.parametrize("k", [5, 40])
def test_runs_in_it(fam, n, prec, k):
    ctx = fam.Context(0)   # a context of its own: nothing larger was allocated before
    X = torch.randn((n, 64), device="cuda", generator=torch.Generator("cuda").manual_seed(n))
    nbr, dist = ctx.knn_graph(X, k, prec)
    ctx.set_knn_pruning(False)
    rn, rd = fam.Context(0).knn_graph(X, k, "fp32")
    assert torch.equal(nbr, rn) and torch.equal(dist, rd)
    T, _ = ctx.emst_exact(X, "bf16x3") if n <= 5000 else (None, None)
    assert T is None or T.u.numel() == n - 1
