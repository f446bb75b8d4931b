"""The whole-solve kernel of small 2-D problems with few blocks (QN_SMALL_GRID): every grid from one
block up gives the solution of the default grid, to the rounding of the norms' summation order.

The products of a row do not depend on the grid, and beta is a minimum and a maximum: the iterates
are equal bit for bit.
"""
import numpy as np
import pytest

from paper_2502_03611_gb300.inputs import manufactured_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [63, 117, 118, 128])
def test_few_blocks(monkeypatch, n):
    import torch

    from paper_2502_03611_gb300 import qn
    qn.load_library()
    f = torch.from_numpy(np.ascontiguousarray(manufactured_problem(n, 2, seed=1)[1])).cuda().reshape(-1)
    outs = []
    for grid in (None, "1", "2", "5"):
        if grid is None:
            monkeypatch.delenv("QN_SMALL_GRID", raising=False)
        else:
            monkeypatch.setenv("QN_SMALL_GRID", grid)
        U = torch.zeros(n * n, dtype=torch.float64, device="cuda")
        res, _ = qn.qn_solve(qn.QnContext(2, n, "fp64"), U, f)
        assert res["status"] == 0, grid
        outs.append((res["iterations"], U))
    for it, U in outs[1:]:
        assert it == outs[0][0] and torch.equal(U, outs[0][1])
