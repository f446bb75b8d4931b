"""FP64 digit products on fields that are not noise, and in passes.

Fields whose digits repeat in every term: the constant row of the Neumann basis on
fields that are constant up to 1e-7, where a sum of d + 1 digit products grows with the number of
terms instead of averaging out. The inverse keeps the bound of any other field: 2 d products, each
within 4 sqrt(n) roundings of its largest terms.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


# halves of 92, 128, 138, 188 and 256 terms; a dense basis with a constant row (Neumann spectral elements, n = 2 E + 1)
@pytest.mark.parametrize("dim,n,sem", [(2, 183, 0), (2, 255, 0), (2, 275, 0), (2, 376, 0), (2, 511, 0), (3, 75, 0),
                                       (2, 255, 2)])
@pytest.mark.parametrize("rows", ["one constant", "one constant each"])
def test_near_constant_fields(dim, n, sem, rows):
    import torch

    from paper_2502_03611_gb300 import qn
    qn.load_library()
    if sem:
        _, S, Si, lam, _ = qn.qn_setup_1d_sem(n, sem, 1.0, qn.QN_BC_NEUMANN)
        ctx = qn.QnContext(dim, n, "fp64", bc="neumann", sem_k=sem)
    else:
        S, Si, lam = qn.qn_setup_1d_eig(n, 1.0 / (n - 1), qn.QN_BC_NEUMANN)
        ctx = qn.QnContext(dim, n, "fp64", bc="neumann")
    rng = np.random.default_rng(n)
    noise = 1.0 + 1e-7 * rng.standard_normal((n,) * dim)
    cs = [0.96668, 0.7071, 0.5557, 0.9999] if rows == "one constant" else [None]
    for c in cs:
        r = noise * (c if c is not None else rng.uniform(0.5, 1.0, size=(n,) * (dim - 1) + (1,)))
        t = torch.from_numpy(r).cuda()
        V = torch.empty_like(t)
        qn.qn_fast_diag_solve(ctx, t, V, 7.0)
        X = r
        for M in (Si, S):
            for a in range(dim):
                X = np.moveaxis(np.tensordot(M, X, axes=([1], [a])), 0, a)
            if M is Si:
                X = X / (sum(lam.reshape([-1 if a == b else 1 for b in range(dim)]) for a in range(dim)) + 7.0)
        err = float(np.abs(V.cpu().numpy() - X).max() / np.abs(X).max())
        assert err <= 2 * dim * 4.0 * np.sqrt(n) * 2.0 ** -52, (c, err)


# values over eight decades and one node a billion times the others, within every row: the digits cut
# each value at 2^-61 of its row's largest
@pytest.mark.parametrize("n,bc", [(190, "dirichlet"), (255, "neumann"), (512, "dirichlet")])
@pytest.mark.parametrize("field", ["wide", "spike"])
def test_rows_of_wide_range(n, bc, field):
    import torch

    from paper_2502_03611_gb300 import qn
    qn.load_library()
    S, Si, lam = qn.qn_setup_1d_eig(n, 1.0 / (n + 1 if bc == "dirichlet" else n - 1), qn.BCS[bc])
    rng = np.random.default_rng(n)
    r = 10.0 ** rng.uniform(-8, 0, (n, n)) * rng.choice([-1.0, 1.0], (n, n))
    if field == "spike":
        r = 1e-9 * rng.standard_normal((n, n))
        r[n // 2, n // 2] = 1.0
    t = torch.from_numpy(r).cuda()
    V = torch.empty_like(t)
    qn.qn_fast_diag_solve(qn.QnContext(2, n, "fp64", bc=bc), t, V, 7.0)
    X = S @ ((Si @ r @ Si.T) / (lam[:, None] + lam[None, :] + 7.0)) @ S.T
    assert np.abs(V.cpu().numpy() - X).max() <= 4 * 4.0 * np.sqrt(n) * 2.0 ** -52 * np.abs(X).max()


@pytest.mark.parametrize("dim,n", [(3, 97), (3, 130), (2, 1001)])
def test_passes_over_the_rows(monkeypatch, dim, n):
    """Digits of a part of the rows at a time (little memory): the same bits."""
    import torch

    from paper_2502_03611_gb300 import qn
    qn.load_library()
    r = torch.from_numpy(np.random.default_rng(n).standard_normal((n,) * dim)).cuda()
    outs = []
    for mb in (None, "1", "7"):
        if mb is None:
            monkeypatch.delenv("QN_DIGIT_MB", raising=False)
        else:
            monkeypatch.setenv("QN_DIGIT_MB", mb)
        V = torch.empty_like(r)
        qn.qn_fast_diag_solve(qn.QnContext(dim, n, "fp64"), r, V, 7.0)
        outs.append(V)
    assert torch.equal(outs[0], outs[1]) and torch.equal(outs[0], outs[2])
