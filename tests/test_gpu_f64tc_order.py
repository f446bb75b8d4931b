"""The FP64 digit products refill the shared-memory tiles of their digits while other tiles are in
use: a tile overwritten before its last reader is done shows as a result that differs from run to
run or from the plain product.

Repeated inverses are compared bit for bit while another stream keeps the memory busy (which
moves the arrival of the tiles), and the first one with numpy's, each of the 2 d products within
4 sqrt(n) roundings of its largest terms.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


# tiles of 64, 32 and 16 columns; one K step of 64 to sixteen (dense products of 1024 terms)
@pytest.mark.parametrize("dim,n,bc", [(3, 50, "dirichlet"), (3, 97, "neumann"), (3, 160, "dirichlet"),
                                      (2, 182, "dirichlet"), (2, 400, "neumann"), (2, 1024, "robin")])
def test_repeated_inverses_are_equal(dim, n, bc):
    import torch

    from paper_2502_03611_gb300 import qn
    qn.load_library()
    h = 1.0 / (n + 1) if bc == "dirichlet" else 1.0 / (n - 1)
    kw = {}
    if bc == "robin":
        S, Si, lam = qn.qn_setup_1d_robin(n, h, 2.0)
        kw["robin_kappa"] = 2.0
    else:
        S, Si, lam = qn.qn_setup_1d_eig(n, h, qn.BCS[bc])
    ctx = qn.QnContext(dim, n, "fp64", bc=bc, **kw)
    r = np.random.default_rng(n).standard_normal((n,) * dim)
    rt = torch.from_numpy(r).cuda()
    V, first = torch.empty_like(rt), None
    noise = torch.empty(1 << 26, dtype=torch.float32, device="cuda")
    side = torch.cuda.Stream()
    for i in range(20):
        with torch.cuda.stream(side):
            for _ in range(i % 4):
                noise.add_(1.0)
        qn.qn_fast_diag_solve(ctx, rt, V, 7.0)
        torch.cuda.synchronize()
        if first is None:
            first = V.clone()
        assert torch.equal(V, first), i
    X = r
    for a in range(dim):
        X = np.moveaxis(np.tensordot(Si, X, axes=([1], [a])), 0, a)
    X = X / (sum(lam.reshape([-1 if a == b else 1 for b in range(dim)]) for a in range(dim)) + 7.0)
    for a in range(dim):
        X = np.moveaxis(np.tensordot(S, X, axes=([1], [a])), 0, a)
    assert np.abs(first.cpu().numpy() - X).max() <= 2 * dim * 4.0 * np.sqrt(n) * 2.0 ** -52 * np.abs(X).max()
