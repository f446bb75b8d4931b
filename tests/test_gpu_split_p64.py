"""Reflection-split products where P / 2 is an odd multiple of 32 (a half ends inside a K step) or
the backward tiles reach past a half, against the dense products.

Both sides stop at a residual of 1e-10 of ||f||, so the solutions agree to 1e-9 of the largest
value, as the dense comparisons at multiples of 128 do; the eigenvalue is the square of the
eigenvector's accuracy (1e-10 against 1e-7). The dense side of P = 704 is left out for its time:
the FP64 residual of the solution is checked there instead, to 1e-10 and its own rounding.
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


def _source(n, seed):
    """Broad-band source without any mirror symmetry, on the device."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.linspace(0.0, 1.0, n + 2, dtype=torch.float64, device="cuda")[1:-1]
    p = x * (1.0 - x) * (1.0 + x)
    f = 40.0 * p[:, None, None] * torch.exp(x)[None, :, None] * p[None, None, :]
    return (f + 0.1 * torch.randn(f.shape, generator=g, dtype=torch.float64, device="cuda")).reshape(-1)


def _solve(qn, n, f, monkeypatch, split, **kw):
    import torch
    monkeypatch.setenv("QN_SPLIT", split)
    ctx = qn.QnContext(3, n, "bf16x3", **kw)
    qn.qn_profile_enable(ctx, True)
    U = torch.zeros(n ** 3, dtype=torch.float64, device="cuda")
    res, _ = qn.qn_solve(ctx, U, f, tol=1e-10, max_it=100)
    prof = qn.qn_profile_read(ctx)
    assert prof["split_products"] == int(split)
    assert res["status"] == 0 and res["rel"] <= 1e-10
    return res, U


@pytest.mark.parametrize("n,bc", [(257, "neumann"), (319, "neumann"), (320, "dirichlet"), (385, "dirichlet"),
                                  (448, "neumann"), (545, "dirichlet"),
                                  (577, "dirichlet")])
def test_split_matches_dense(qn, monkeypatch, n, bc):
    f = _source(n, n)
    kw = dict(bc=bc, lam=3.0) if bc == "neumann" else dict(bc=bc)
    (r1, u1), (r0, u0) = (_solve(qn, n, f, monkeypatch, s, **kw) for s in ("1", "0"))
    assert abs(r1["iterations"] - r0["iterations"]) <= 1
    assert float((u1 - u0).abs().max()) <= 1e-9 * float(u0.abs().max())


def test_split_reaches_past_a_half(qn, monkeypatch):
    """P = 704: three backward tiles of 128 rows over a half of 352."""
    n = 641
    f = _source(n, 1)
    _, U = _solve(qn, n, f, monkeypatch, "1")
    u = U.reshape(n, n, n)
    r = 6.0 * u
    r[1:] -= u[:-1]
    r[:-1] -= u[1:]
    r[:, 1:] -= u[:, :-1]
    r[:, :-1] -= u[:, 1:]
    r[:, :, 1:] -= u[:, :, :-1]
    r[:, :, :-1] -= u[:, :, 1:]
    r *= float((n + 1) ** 2)
    r += u ** 3
    r = r.reshape(-1) - f
    # the eight FP64 operations above round at up to 2^-53 of 6 |u| / h^2 each
    rounding = 8 * 2.0 ** -53 * 6.0 * (n + 1) ** 2 * float(U.norm() / f.norm())
    assert float(r.norm() / f.norm()) <= 1e-10 + rounding


def test_split_with_potential(qn, monkeypatch):
    """Example 1 of Sec. 6.3 (Neumann, potential) on 258^3."""
    import torch
    n = 258
    u, f, v, h = I.ex1_problem(n)
    U0 = u + I.ex1_perturbation(n, 4, 0.1)
    sols = []
    for split in ("1", "0"):
        monkeypatch.setenv("QN_SPLIT", split)
        ctx = qn.QnContext(3, n, "bf16x3", lam=I.EX1_A, b=I.EX1_B, bc="neumann", length=2.0, potential=v)
        U = torch.from_numpy(np.ascontiguousarray(U0)).cuda().reshape(-1).clone()
        res, _ = qn.qn_solve(ctx, U, torch.from_numpy(np.ascontiguousarray(f)).cuda().reshape(-1), tol=1e-10,
                             max_it=300)
        assert res["status"] == 0
        sols.append((res["iterations"], U))
    assert abs(sols[0][0] - sols[1][0]) <= 1
    assert float((sols[0][1] - sols[1][1]).abs().max()) <= 1e-9 * float(sols[1][1].abs().max())


def test_split_eigenproblem(qn, monkeypatch):
    import torch
    n = 257
    v, h, x = I.ex2_problem(n)
    U0 = I.ex2_start(n, seed=2)
    outs = []
    for split in ("1", "0"):
        monkeypatch.setenv("QN_SPLIT", split)
        ctx = qn.QnContext(3, n, "bf16x3", lam=0.0, b=I.EX2_ALPHA, bc="dirichlet", length=I.EX2_LENGTH, potential=v)
        qn.qn_profile_enable(ctx, True)
        U = torch.from_numpy(np.ascontiguousarray(U0)).cuda().reshape(-1).clone()
        res, _ = qn.qn_eig_solve(ctx, U)
        assert res["status"] == 0 and qn.qn_profile_read(ctx)["split_products"] == int(split)
        outs.append((res["lambda"], U))
    assert outs[0][0] == pytest.approx(outs[1][0], rel=1e-10)
    assert float((outs[0][1] - outs[1][1]).abs().max()) <= 1e-7 * float(outs[1][1].abs().max())


def test_refusals_stand(qn):
    """What needs P a multiple of 128 is refused at other sizes, split products or not."""
    with pytest.raises(RuntimeError, match="BF16X6"):
        qn.QnContext(3, 258, "bf16x6")
    ctx = qn.QnContext(3, 258, "bf16x3")
    with pytest.raises(RuntimeError):
        qn.qn_set_escalation(ctx, 1e-3)
    with pytest.raises(RuntimeError):
        qn.qn_set_fused_residual(ctx, True)
