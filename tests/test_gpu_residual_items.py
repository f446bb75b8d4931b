"""Work items of the split residual kernels: planes per item chosen from the sizes, and only the
tiles that hold grid points visited (the padding is zeroed apart).

The residual of a node and the extremes behind beta do not depend on how the planes are cut into
items, so three iterations give the same U bit for bit whatever the cut; the residual norms are
sums in another order (n^3 terms in FP32 with a carry per thread: 1e-6 relative).
"""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qn():
    import torch  # noqa: F401
    from paper_2502_03611_gb300 import build as B
    from paper_2502_03611_gb300 import qn as Q
    B.build()
    Q.load_library()
    return Q


@pytest.mark.parametrize("n,bc,split", [(65, "dirichlet", "1"), (97, "neumann", "1"), (128, "dirichlet", "1"),
                                        (129, "neumann", "1"), (161, "dirichlet", "1"), (192, "dirichlet", "0"),
                                        (97, "dirichlet", "0"), (257, "neumann", "1"), (289, "dirichlet", "1")])
def test_cut_into_items_does_not_change_the_result(qn, monkeypatch, n, bc, split):
    import torch
    g = torch.Generator(device="cuda").manual_seed(n)
    f = torch.randn(n ** 3, generator=g, dtype=torch.float64, device="cuda") + 20.0
    U0 = torch.randn(n ** 3, generator=g, dtype=torch.float64, device="cuda")
    monkeypatch.setenv("QN_SPLIT", split)
    outs = []
    for zc in (None, "1", "32", "4096"):
        if zc is None:
            monkeypatch.delenv("QN_RES_ZC", raising=False)
        else:
            monkeypatch.setenv("QN_RES_ZC", zc)
        ctx = qn.QnContext(3, n, "bf16x3", bc=bc, lam=2.0 if bc == "neumann" else 0.0)
        U = U0.clone()
        _, hist = qn.qn_solve(ctx, U, f, tol=1e-15, max_it=3, history_len=4)
        outs.append((U, [h["rel"] for h in hist]))
    for U, rel in outs[1:]:
        assert torch.equal(U, outs[0][0])
        assert rel == pytest.approx(outs[0][1], rel=1e-6)
