"""Passes of the eigenvalue iteration over tiles shaped by the grid size (pass 1) and flat mirror
pairs (pass 2): the BF16X3 solve against the FP64 one.

Both stop at a relative residual of 1e-10; the eigenvalue, second order in the eigenvector's
error, agrees to 1e-9 and the normalised eigenvector to 1e-7, as against the oracle.
"""
import numpy as np
import pytest

from paper_2502_03611_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qn():
    import torch  # noqa: F401
    from paper_2502_03611_gb300 import build as B
    from paper_2502_03611_gb300 import qn as Q
    B.build()
    Q.load_library()
    return Q


@pytest.mark.parametrize("n,bc", [(3, "dirichlet"), (23, "dirichlet"), (25, "neumann"), (33, "dirichlet"),
                                  (50, "neumann"), (65, "neumann"), (66, "dirichlet"), (97, "neumann"),
                                  (104, "dirichlet"), (127, "dirichlet"), (128, "neumann"), (130, "dirichlet")])
def test_tile_shapes(qn, n, bc):
    import torch
    v, h, x = I.ex2_problem(n)
    U0 = I.ex2_start(n, seed=n)
    outs = []
    for prec in ("bf16x3", "fp64"):
        ctx = qn.QnContext(3, n, prec, lam=1.0 if bc == "neumann" else 0.0, b=I.EX2_ALPHA, bc=bc,
                           length=I.EX2_LENGTH, potential=v)
        U = torch.from_numpy(np.ascontiguousarray(U0)).cuda().reshape(-1).clone()
        res, _ = qn.qn_eig_solve(ctx, U)
        assert res["status"] == 0, (prec, res)
        outs.append((res["lambda"], U))
    assert outs[0][0] == pytest.approx(outs[1][0], rel=1e-9)
    assert float((outs[0][1] - outs[1][1]).abs().max()) <= 1e-7 * float(outs[1][1].abs().max())
