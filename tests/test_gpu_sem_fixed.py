"""The integer banded sums of the split spectral element solves: the residual norm of the first
updated iterate against the FP64 kernel's, over the degrees."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qn():
    from paper_2502_03611_gb300 import qn as q
    q.load_library()
    return q


# every band width up to the widest; rows in groups of four with remainders
@pytest.mark.parametrize("dim,k,E,bc", [(2, 1, 40, "dirichlet"), (3, 2, 12, "neumann"), (3, 3, 9, "dirichlet"),
                                        (2, 4, 30, "neumann"), (3, 5, 7, "dirichlet"), (3, 8, 4, "neumann"),
                                        (2, 10, 13, "dirichlet"), (3, 10, 3, "neumann"), (2, 11, 6, "dirichlet"),
                                        (2, 16, 4, "neumann")])
@pytest.mark.parametrize("pot", [False, True])
def test_residual_norm_of_the_next_iterate(qn, dim, k, E, bc, pot):
    import torch
    n = E * k - 1 if bc == "dirichlet" else E * k + 1
    rng = np.random.default_rng(n + k)
    f = torch.from_numpy(rng.standard_normal((n,) * dim) * 50.0).cuda()
    U0 = torch.from_numpy(rng.standard_normal((n,) * dim)).cuda()
    v = rng.random(n) * 3.0 if pot else None
    kw = dict(lam=2.0, b=1.0, bc=bc, potential=v, sem_k=k)
    ctx, ref = qn.QnContext(dim, n, "bf16x3", **kw), qn.QnContext(dim, n, "fp64", **kw)
    U = U0.clone()
    res, hist = qn.qn_solve(ctx, U, f, tol=0.0, max_it=1, beta=500.0, history_len=2)
    R = torch.empty_like(U)
    want = qn.qn_residual(ref, U, f, R)
    assert res["iterations"] == 1
    # both sums carry a few roundings of the largest terms: max|U| times the largest row sum of H
    H = qn.qn_setup_1d_sem(n, k, 1.0, qn.BCS[bc])[0]
    scale = float(U.abs().max()) * np.abs(H).sum(axis=1).max() * dim
    tol = 2.0 ** -53 * 3 * (2 * k + 1) * scale * n ** (dim / 2)
    assert abs(hist[1]["res_norm"] - want["res_norm"]) <= tol + 1e-14 * want["res_norm"]
    assert hist[1]["fu_max"] == pytest.approx(want["fu_max"], rel=1e-15)
    assert hist[1]["fu_min"] == pytest.approx(want["fu_min"], rel=1e-15, abs=1e-15)


@pytest.mark.parametrize("scale", [2.0 ** 60, 2.0 ** -70])
def test_values_out_of_the_fixed_point_range(qn, scale):
    """A linear problem scaled by a power of two: the FP64 kernel takes over and the solution scales."""
    import torch
    n, k = 31, 4
    f = torch.from_numpy(np.random.default_rng(0).standard_normal((n, n, n))).cuda()
    out = []
    for s in (1.0, scale):
        ctx = qn.QnContext(3, n, "bf16x3", lam=1.0, b=0.0, sem_k=k)
        U = torch.zeros_like(f)
        res, _ = qn.qn_solve(ctx, U, f * s, tol=1e-10)
        assert res["status"] == 0
        out.append(U / s)
    assert float((out[0] - out[1]).abs().max()) <= 1e-8 * float(out[0].abs().max())
