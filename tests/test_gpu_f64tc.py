"""The FP64 mode products on the tensor cores (exact integer digits), through the shifted
inverse: sizes at the edges of the tiles, K steps, sums and dispatch rule, every boundary type
and basis, magnitudes across the FP64 range, and non-finite inputs."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qn():
    from paper_2502_03611_gb300 import qn as q
    q.load_library()
    return q


def _numpy_inverse(r, S, Si, lam, shift):
    X, d = r, r.ndim
    for a in range(d):
        X = np.moveaxis(np.tensordot(Si, X, axes=([1], [a])), 0, a)
    X = X / (sum(lam.reshape([-1 if a == b else 1 for b in range(d)]) for a in range(d)) + shift)
    for a in range(d):
        X = np.moveaxis(np.tensordot(S, X, axes=([1], [a])), 0, a)
    return X


def _inverse(qn, ctx, r, shift):
    import torch
    t = torch.from_numpy(np.ascontiguousarray(r)).cuda()
    V = torch.full_like(t, np.nan)
    qn.qn_fast_diag_solve(ctx, t, V, shift)
    torch.cuda.synchronize()
    return V.cpu().numpy()


def _tol(n, dim):
    """2 d products, each within 4 sqrt(n) roundings of its largest terms (numpy's sums)."""
    return 2 * dim * 4.0 * np.sqrt(n) * 2.0 ** -52


def _basis(qn, kind, n):
    if kind == "dirichlet":
        return qn.qn_setup_1d_eig(n), dict()
    if kind == "neumann":
        return qn.qn_setup_1d_eig(n, 1.0 / (n - 1), qn.QN_BC_NEUMANN), dict(bc="neumann")
    if kind == "robin":
        return qn.qn_setup_1d_robin(n, 1.0 / (n - 1), 2.0), dict(bc="robin", robin_kappa=2.0)
    _, S, Si, lam, _ = qn.qn_setup_1d_sem(n, 3)
    return (S, Si, lam), dict(sem_k=3)


# 3-D from the first size on this path (50); halves of 32, 33, 64, 65 rows and 128 / 129 terms;
# 2-D from its first size (182); sums of more than 128 and 256 terms; two sums per half
@pytest.mark.parametrize("dim,n,kind", [
    (3, 49, "dirichlet"), (3, 50, "dirichlet"), (3, 63, "dirichlet"), (3, 64, "neumann"), (3, 65, "dirichlet"),
    (3, 127, "neumann"), (3, 128, "dirichlet"), (3, 129, "dirichlet"), (3, 131, "neumann"),
    (3, 53, "sem"), (3, 66, "robin"),
    (2, 181, "dirichlet"), (2, 182, "dirichlet"), (2, 255, "neumann"), (2, 256, "dirichlet"), (2, 257, "dirichlet"),
    (2, 300, "neumann"), (2, 512, "dirichlet"), (2, 513, "neumann"), (2, 1024, "dirichlet"), (2, 1024, "neumann"),
    (2, 254, "sem"), (2, 257, "robin"), (2, 518, "sem"), (2, 1023, "robin")])
def test_inverse_matches_numpy(qn, dim, n, kind):
    (S, Si, lam), kw = _basis(qn, kind, n)
    rng = np.random.default_rng(n)
    r = rng.standard_normal((n,) * dim)
    r += 20.0 * np.sin(np.arange(n) / n)          # a smooth part along x
    ctx = qn.QnContext(dim, n, "fp64", **kw)
    V = _inverse(qn, ctx, r, 7.0)
    ref = _numpy_inverse(r, S, Si, lam, 7.0)
    assert np.abs(V - ref).max() <= _tol(n, dim) * np.abs(ref).max()


@pytest.mark.parametrize("scale", [1e-300, 1e-160, 1e200, 1e290])
def test_inverse_over_the_fp64_range(qn, scale):
    """Powers of two scale the result exactly while it stays normal; rows of very different size."""
    n = 200
    rng = np.random.default_rng(1)
    r = rng.standard_normal((n, n)) * 10.0 ** rng.integers(-8, 8, size=(n, 1))
    r[17] = 0.0
    ctx = qn.QnContext(2, n, "fp64")
    s = 2.0 ** np.floor(np.log2(scale))
    V1, Vs = _inverse(qn, ctx, r, 3.0), _inverse(qn, ctx, r * s, 3.0)
    ok = np.abs(V1) * s > 1e-305
    assert np.array_equal(Vs[ok], (V1 * s)[ok]) and np.all(np.isfinite(Vs))
    assert np.abs(Vs / s - V1).max() <= 1e-4 * np.abs(V1).max()


def test_inverse_of_zero_and_subnormals(qn):
    n = 190
    ctx = qn.QnContext(2, n, "fp64")
    assert not _inverse(qn, ctx, np.zeros((n, n)), 3.0).any()
    r = np.full((n, n), 5e-324)
    assert np.all(np.isfinite(_inverse(qn, ctx, r, 3.0)))


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
def test_non_finite_values_propagate(qn, value):
    """One bad entry reaches every output, as in a sum of products."""
    n = 200
    ctx = qn.QnContext(2, n, "fp64")
    r = np.ones((n, n))
    r[3, 70] = value
    with np.errstate(invalid="ignore"):
        S, Si, lam = qn.qn_setup_1d_eig(n)
        ref = _numpy_inverse(r, S, Si, lam, 3.0)
    V = _inverse(qn, ctx, r, 3.0)
    assert not np.isfinite(V).any() and not np.isfinite(ref).any()


@pytest.mark.parametrize("dim,n,shift", [(2, 200, 1e-300), (3, 50, 1e300), (2, 200, 0.0)])
def test_divisor_range(qn, dim, n, shift):
    """The integer quotient against divisors across the FP64 range."""
    r = np.random.default_rng(5).standard_normal((n,) * dim)
    S, Si, lam = qn.qn_setup_1d_eig(n)
    V = _inverse(qn, qn.QnContext(dim, n, "fp64"), r, shift)
    ref = _numpy_inverse(r, S, Si, lam, shift)
    assert np.abs(V - ref).max() <= _tol(n, dim) * np.abs(ref).max()


def test_solve_matches_oracle_and_graph(qn):
    """A 3-D FP64 solve on this path: the oracle's iterates, and the same bits from graph replay."""
    import torch

    import oracle as O
    from paper_2502_03611_gb300.inputs import manufactured_problem
    n = 65
    _, f = manufactured_problem(n, 3, seed=3)
    ft = torch.from_numpy(f).cuda()
    ctx = qn.QnContext(3, n, "fp64")
    out = []
    for graph in (False, True):
        U = torch.zeros_like(ft)
        res, _ = qn.qn_solve(ctx, U, ft, graph=graph)
        assert res["status"] == 0
        out.append((U.cpu().numpy(), res["iterations"]))
    Uo, hist, ok = O.qn_solve(f)
    assert ok and out[0][1] == len(hist) - 1 == out[1][1]
    assert np.array_equal(out[0][0], out[1][0])
    assert np.abs(out[0][0] - Uo).max() <= 1e-12 * np.abs(Uo).max()
