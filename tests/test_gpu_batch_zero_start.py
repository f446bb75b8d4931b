"""Iteration 0 of the batched systems from a zero start (F = -f, no FP64 stencil) against the same
iteration through the general path.

Start values of 1e-300 take the general path and change no bit of it: they vanish in every sum
with the O(1) sources and in the first update. So the solutions and the residuals are equal bit
for bit, whatever part of a row is zero.
"""
import numpy as np
import pytest

from paper_2502_03611_gb300.inputs import coupled_problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qn():
    import torch  # noqa: F401
    from paper_2502_03611_gb300 import build as B
    from paper_2502_03611_gb300 import qn as Q
    B.build()
    Q.load_library()
    return Q


def _start(n, kind):
    import torch
    u = torch.zeros(n, n, dtype=torch.float64, device="cuda")
    if kind == "minus zero":
        u = -u
    elif kind == "tiny":
        u += 1e-300
    elif kind == "tiny right":
        u[:, (2 * n) // 3:] = 1e-300
    elif kind == "tiny left":
        u[:, : n // 3 + 1] = 1e-300
    return u.reshape(-1)


def test_zero_start_matches_general_path(qn):
    import torch
    specs = [(1, 0.2, 1.0, 6), (31, 0.3, 0.5, 1), (65, -0.9, 7.0, 2), (100, 0.5, 2.0, 4), (127, 0.0, 0.3, 5)]
    outs = {}
    for kind in ("tiny", "zero", "minus zero", "tiny right", "tiny left"):
        insts = []
        for (n, alpha, D, seed) in specs:
            _, _, f1, f2 = coupled_problem(n, alpha, D, seed)
            insts.append({"n": n, "alpha": alpha, "D": D, "U": _start(n, kind), "V": _start(n, kind),
                          "f1": torch.from_numpy(f1.reshape(-1)).cuda(), "f2": torch.from_numpy(f2.reshape(-1)).cuda()})
            assert np.abs(f1).min() > 1e-200 and np.abs(f2).min() > 1e-200
        batch = qn.QnBatch(insts)
        rc, res = batch.solve(sync_every=3)
        assert rc == 0
        outs[kind] = [(i["U"], i["V"], r["iterations"], r["rel"]) for i, r in zip(insts, res)]
    for kind, rows in outs.items():
        for a, b in zip(rows, outs["tiny"]):
            assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1]) and a[2:] == b[2:], kind
