"""Performance cases: what a user of this library has it do, through its public entry points.

Each case is one call on the GPU, from the smallest solve (latency) to the largest (memory and
tensor-core throughput), with sizes from the library's tests and benchmark:

* solve2d     2-D finite differences in FP64 (the default precision): the 63^2 Dirichlet latency
              workload, and Example 1 of Sec. 6.2 (Neumann data) on an odd size of the paper's range.
* solve3d     3-D Dirichlet solves from the zero start: the plain FP64 workload, the split-precision
              headline, and the six-product level on random-field sources (data generation for a
              learned start).
* inverse3d   one application of the shifted inverse in FP64 (the operator as a preconditioner).
* residual3d  one FP64 residual with its statistics (checking a field that came from elsewhere).
* ex1         the three-dimensional Example 1 of Sec. 6.3: Neumann data and a potential.
* eig         the nonlinear eigenproblem of Sec. 6.3, Example 2.
* sem         a Q^k spectral element solve (Sec. 3.1).
* batch       many coupled two-component 2-D systems of mixed sizes in one batch (Sec. 4.3).
* net         loss and gradients of the warm-start network on one training batch.

`exact` computes what `run` returns in 64 bits with torch and numpy alone.
"""
import math

import numpy as np
import torch

from paper_2502_03611_gb300 import qn

TOL = 1e-10
DEV = "cuda"


def listed():
    return [
        # a parameter sweep of small 2-D solves: launches and barriers count, not arithmetic
        {"name": "solve2d_fp64_63", "kind": "solve2d", "n": 63, "bc": "dirichlet"},
        # the paper's 2-D Neumann example at about its largest mesh
        {"name": "solve2d_neumann_fp64_1001", "kind": "solve2d", "n": 1001, "bc": "neumann"},
        # the plain FP64 solve, the default precision of a context
        {"name": "solve3d_fp64_255", "kind": "solve3d", "n": 255, "precision": "fp64", "source": "series"},
        # the FP64 inverse alone, on a size that no tile divides
        {"name": "inverse3d_fp64_200", "kind": "inverse3d", "n": 200},
        # the FP64 residual of a given field
        {"name": "residual3d_fp64_400", "kind": "residual3d", "n": 400},
        # the headline: the split-precision solve of the model problem
        {"name": "solve3d_bf16x3_511", "kind": "solve3d", "n": 511, "precision": "bf16x3", "source": "series"},
        # nearly linear solves on random-field sources at the six-product level
        {"name": "solve3d_grf_bf16x6_255", "kind": "solve3d", "n": 255, "precision": "bf16x6", "source": "grf"},
        # Neumann data and a potential; the padded grid is not a multiple of 128
        {"name": "ex1_bf16x3_400", "kind": "ex1", "n": 400},
        # several hundred cheap iterations
        {"name": "eig_bf16x3_100", "kind": "eig", "n": 100},
        # spectral elements: a banded FP64 operator and dense products
        {"name": "sem_q4_bf16x3_255", "kind": "sem", "n": 255, "k": 4},
        # the batched workload: uneven sizes, grouped launches
        {"name": "batch_256", "kind": "batch", "count": 256, "nmin": 63, "nmax": 511},
        # one training batch of the warm-start network
        {"name": "net_grad_64_b8", "kind": "net", "G": 64, "B": 8},
    ]


def _log(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["solve2d", "solve2d", "solve3d", "solve3d", "solve3d", "inverse3d", "residual3d",
                       "ex1", "eig", "sem", "batch", "net"])
    if kind == "solve2d":
        return {"kind": kind, "n": _log(rng, 15, 1001), "bc": rng.choice(["dirichlet", "neumann"])}
    if kind == "solve3d":
        p = rng.choice(["fp64", "bf16x3", "bf16x6"])
        if p == "fp64":
            return {"kind": kind, "n": _log(rng, 24, 250), "precision": p, "source": "series"}
        if p == "bf16x3":
            return {"kind": kind, "n": _log(rng, 40, 510), "precision": p, "source": rng.choice(["series", "grf"])}
        P = 128 * rng.randint(1, 4)     # the six-product level wants 64 ceil(n/64) a multiple of 128
        return {"kind": kind, "n": rng.randint(P - 63, P - 2), "precision": p, "source": "grf"}
    if kind == "inverse3d":
        return {"kind": kind, "n": _log(rng, 24, 255)}
    if kind == "residual3d":
        return {"kind": kind, "n": _log(rng, 40, 399)}
    if kind == "ex1":
        return {"kind": kind, "n": _log(rng, 40, 300)}
    if kind == "eig":
        return {"kind": kind, "n": _log(rng, 32, 99)}
    if kind == "sem":
        k = rng.randint(2, 6)
        return {"kind": kind, "n": k * rng.randint(40 // k, 254 // k) - 1, "k": k}
    if kind == "batch":
        lo = rng.choice([31, 63, 100])
        return {"kind": kind, "count": _log(rng, 16, 200), "nmin": lo, "nmax": rng.randint(200, 511)}
    return {"kind": kind, "G": rng.randint(32, 63), "B": rng.randint(1, 8)}


# ---------------------------------------------------------------------------------------------
# inputs, made on the GPU from the seed
# ---------------------------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator()
    g.manual_seed(int(seed))
    return g


def _grid(n):
    return torch.arange(1, n + 1, dtype=torch.float64, device=DEV) / (n + 1)


def _sines(n, kmax):
    k = torch.arange(1, kmax + 1, dtype=torch.float64, device=DEV)
    return torch.sin(math.pi * k[:, None] * _grid(n)[None, :])


def _series(coef, n):
    """sum_k coef[k] prod_a sin(k_a pi x_a) on the n^dim interior nodes, one axis at a time."""
    B, out = _sines(n, coef.shape[0]), coef
    for axis in range(coef.ndim):
        out = torch.movedim(torch.tensordot(B, out, dims=([0], [axis])), 0, axis)
    return out.contiguous()


def _ksq(kmax, dim):
    k = torch.arange(1, kmax + 1, dtype=torch.float64, device=DEV) ** 2
    return sum(k.reshape([-1 if a == b else 1 for b in range(dim)]) for a in range(dim)).expand((kmax,) * dim)


def _manufactured(n, dim, g):
    """u* and -Lap u* of a sine series with N(0, 1) coefficients on the low modes."""
    kmax = 4 if dim == 2 else 6
    c = 0.1 * torch.randn((kmax,) * dim, generator=g, dtype=torch.float64).to(DEV)
    c[(0,) * dim] += 1.0
    return _series(c, n), _series(c * math.pi ** 2 * _ksq(kmax, dim), n)


def _source(case, seed, dim):
    n, g = case["n"], _gen(seed)
    if case.get("source") == "grf":
        xi = torch.randn((32,) * 3, generator=g, dtype=torch.float64).to(DEV)
        f = _series(xi / (1.0 + _ksq(32, 3)), n)
        return f / torch.sqrt(torch.mean(f * f))
    u, lap = _manufactured(n, dim, g)
    return lap + u ** 3


def _rough(n, seed):
    """A residual as the inverse meets it: smooth low modes and noise at every scale."""
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    return _manufactured(n, 3, _gen(seed))[1] + torch.rand((n,) * 3, generator=g, dtype=torch.float64, device=DEV)


def _poly(x, g, dim):
    """A random polynomial of degree 4 per axis, its largest value on the nodes 1."""
    c = torch.rand((5,) * dim, generator=g, dtype=torch.float64).to(DEV) * 2 - 1
    V = torch.stack([x ** i for i in range(5)])
    for axis in range(dim):
        c = torch.movedim(torch.tensordot(V, c, dims=([0], [axis])), 0, axis)
    return (c / c.abs().max()).contiguous()


def _potential_1d(x):
    return 100.0 * torch.sin(0.25 * math.pi * x) ** 2 + x * x


def _sum3(v):
    return v[:, None, None] + v[None, :, None] + v[None, None, :]


def _ex2d1(n):
    x = torch.linspace(-1.0, 1.0, n, dtype=torch.float64, device=DEV)
    u = torch.cos(2 * math.pi * x)[:, None] * torch.cos(math.pi * x)[None, :]
    return x, u, (5 * math.pi ** 2 + 1.0) * u + u ** 3


def _ex1(n, seed):
    x = torch.linspace(-1.0, 1.0, n, dtype=torch.float64, device=DEV)
    v, u = _potential_1d(x), _sum3(torch.cos(math.pi * x))
    f = (math.pi ** 2 + 10.0) * u + 10.0 * u ** 3 + _sum3(v) * u
    return v, f, u + 0.1 * _poly(x, _gen(seed), 3)


def _ex2(n, seed):
    h = 16.0 / (n + 1)
    x = -8.0 + h * torch.arange(1, n + 1, dtype=torch.float64, device=DEV)
    g = torch.cos(math.pi * x / 16.0)
    start = g[:, None, None] * g[None, :, None] * g[None, None, :]
    return _potential_1d(x), h, start * (1.0 + 0.1 * _poly(x / 8.0, _gen(seed), 3))


def _sem_nodes(n, k):
    xi = np.concatenate([[-1.0], np.sort(np.polynomial.legendre.Legendre.basis(k).deriv().roots().real), [1.0]])
    E = (n + 1) // k
    x = np.concatenate([(e + 0.5 * (1.0 + xi[:-1])) / E for e in range(E)])[1:]
    return xi, E, torch.from_numpy(x).to(DEV)


def _sem_source(case, seed):
    """Source of a smooth manufactured solution at the Gauss-Lobatto nodes."""
    n, g = case["n"], _gen(seed)
    x = _sem_nodes(n, case["k"])[2]
    c = 0.1 * torch.randn((6,) * 3, generator=g, dtype=torch.float64).to(DEV)
    c[0, 0, 0] += 1.0
    B = torch.sin(math.pi * torch.arange(1, 7, dtype=torch.float64, device=DEV)[:, None] * x[None, :])
    ev = lambda t: torch.einsum("abc,az,by,cx->zyx", t, B, B, B)  # noqa: E731
    u = ev(c)
    return (ev(c * math.pi ** 2 * _ksq(6, 3)) + u ** 3).contiguous()


def _system_sizes(case):
    """The grid sizes that the instances take in turn: 2^j - 1, or odd ones between."""
    sizes = [m for m in (31, 63, 127, 255, 511) if case["nmin"] <= m <= case["nmax"]]
    if case["nmax"] not in sizes:
        sizes += [case["nmin"], (case["nmin"] + case["nmax"]) // 2, case["nmax"]]
    return sizes


def _systems(case, seed):
    """Parameters and sources of the coupled instances."""
    g = _gen(seed)
    sizes, out = _system_sizes(case), []
    for i in range(case["count"]):
        a, d = torch.rand(2, generator=g, dtype=torch.float64).tolist()
        n, alpha, D = sizes[i % len(sizes)], a, 0.1 + 9.9 * d
        (u, lu), (v, lv) = _manufactured(n, 2, g), _manufactured(n, 2, g)
        out.append((n, alpha, D, lu + u ** 3 + alpha * v, D * lv + v ** 3 - alpha * u))
    return out


def _net_params(C, M, L, g):
    """Random weights at the scale of a freshly initialised network, in the flat parameter order."""
    parts = [torch.randn(C, generator=g), torch.zeros(C)]
    for _ in range(L):
        parts += [torch.randn(M ** 3 * C * C, generator=g) / C, torch.randn(C * C, generator=g) / math.sqrt(C),
                  torch.zeros(C)]
    return torch.cat(parts + [torch.randn(C, generator=g) / math.sqrt(C), torch.zeros(1)]).float()


def _net_data(case, seed):
    G, B, g = case["G"], case["B"], _gen(seed)
    p = _net_params(32, 6, 4, g)
    f = torch.stack([_series(torch.randn((16,) * 3, generator=g, dtype=torch.float64).to(DEV) / (1.0 + _ksq(16, 3)), G)
                     for _ in range(B)])
    f /= torch.sqrt(torch.mean(f * f))
    t = torch.stack([_series(torch.randn((6,) * 3, generator=g, dtype=torch.float64).to(DEV) / (1.0 + _ksq(6, 3)), G)
                     for _ in range(B)])
    t /= torch.sqrt(torch.mean(t * t))
    return p, f.float().contiguous(), t.float().contiguous()


# ---------------------------------------------------------------------------------------------
# what a program keeps (prepare) and one call (run)
# ---------------------------------------------------------------------------------------------
def prepare(case, seed):
    kind, n = case["kind"], case.get("n", 0)
    s = {"kind": kind}
    if kind == "solve2d":
        if case["bc"] == "dirichlet":
            f, ctx = _source(case, seed, 2), qn.QnContext(2, n, "fp64")
            start = torch.zeros_like(f)
        else:
            x, u, f = _ex2d1(n)
            ctx = qn.QnContext(2, n, "fp64", lam=1.0, b=1.0, bc="neumann", length=2.0)
            start = u + 0.1 * _poly(x, _gen(seed), 2)
        s.update(ctx=ctx, f=f, start=start, U=torch.empty_like(f), graph=False)
    elif kind == "solve3d":
        f = _source(case, seed, 3)
        s.update(ctx=qn.QnContext(3, n, case["precision"]), f=f, start=None, U=torch.empty_like(f),
                 graph=case["precision"] != "fp64")
    elif kind == "inverse3d":
        r = _rough(n, seed)
        s.update(ctx=qn.QnContext(3, n, "fp64"), r=r, V=torch.empty_like(r))
    elif kind == "residual3d":
        f = _source(case, seed, 3)
        u = _manufactured(n, 3, _gen(seed + 1))[0]
        s.update(ctx=qn.QnContext(3, n, "fp64"), U=u, f=f, R=torch.empty_like(u))
    elif kind == "ex1":
        v, f, start = _ex1(n, seed)
        ctx = qn.QnContext(3, n, "bf16x3", lam=10.0, b=10.0, bc="neumann", length=2.0, potential=v.cpu().numpy())
        s.update(ctx=ctx, f=f, start=start, U=torch.empty_like(f), graph=True)
    elif kind == "eig":
        v, _, start = _ex2(n, seed)
        ctx = qn.QnContext(3, n, "bf16x3", b=1600.0, length=16.0, potential=v.cpu().numpy())
        s.update(ctx=ctx, start=start, U=torch.empty_like(start))
    elif kind == "sem":
        f = _sem_source(case, seed)
        s.update(ctx=qn.QnContext(3, n, "bf16x3", sem_k=case["k"]), f=f, start=None, U=torch.empty_like(f), graph=True)
    elif kind == "batch":
        inst, at = _systems(case, seed), 0
        off = []
        for m, *_ in inst:      # all iterates in one slab, so that one fill resets them
            off.append(at)
            at += 2 * (-(-m * m // 32) * 32)
        slab = torch.zeros(at, dtype=torch.float64, device=DEV)
        views = [(slab[o:o + m * m].view(m, m), slab[o + -(-m * m // 32) * 32:][:m * m].view(m, m))
                 for o, (m, *_) in zip(off, inst)]
        batch = qn.QnBatch([{"n": m, "alpha": a, "D": d, "U": u, "V": v, "f1": f1, "f2": f2}
                            for (m, a, d, f1, f2), (u, v) in zip(inst, views)])
        s.update(batch=batch, slab=slab)
    else:
        p, f, t = _net_data(case, seed)
        net = qn.QnNet(case["G"], max_batch=case["B"])
        net.set_params(p.numpy())
        s.update(net=net, f=f, t=t, B=case["B"], grads=torch.empty(net.nparams, dtype=torch.float32, device=DEV))
    torch.cuda.synchronize()
    return s


def run(s):
    kind = s["kind"]
    if kind in ("solve2d", "solve3d", "ex1", "sem"):
        if s["start"] is None:
            s["U"].zero_()
        else:
            s["U"].copy_(s["start"])
        res, _ = qn.qn_solve(s["ctx"], s["U"], s["f"], tol=TOL, graph=s["graph"])
        return {"U": s["U"], "iterations": res["iterations"]}
    if kind == "inverse3d":
        qn.qn_fast_diag_solve(s["ctx"], s["r"], s["V"], 3.0)
        return s["V"]
    if kind == "residual3d":
        st = qn.qn_residual(s["ctx"], s["U"], s["f"], s["R"])
        return {"R": s["R"], "stats": [st["res_norm"], st["f_norm"], st["fu_min"], st["fu_max"], st["beta"]]}
    if kind == "eig":
        s["U"].copy_(s["start"])
        res, _ = qn.qn_eig_solve(s["ctx"], s["U"], tol=TOL, graph=True)
        return {"U": s["U"], "lambda": res["lambda"]}
    if kind == "batch":
        s["slab"].zero_()
        _, res = s["batch"].solve(tol=TOL)
        return {"UV": s["slab"], "iterations": np.array([r["iterations"] for r in res])}
    loss = s["net"].gradients(s["f"], s["t"], s["B"], s["grads"])
    return {"loss": loss, "grads": s["grads"]}


def work(case):
    """Bytes: the inputs read and the outputs written once per iteration (the stop test and beta need
    the whole iterate). Flops: the mode products with the reflection symmetry used (half of 2 n^(d+1)
    each), for spectral elements in full, times a typical iteration count."""
    kind, n = case["kind"], case.get("n", 0)
    if kind == "solve2d":
        it = 7 if case["bc"] == "dirichlet" else 10
        return {"bytes": it * 24 * n ** 2, "flops": it * 4 * n ** 3}
    if kind == "solve3d":
        it = 3 if case["source"] == "grf" else 12
        return {"bytes": it * 24 * n ** 3, "flops": it * 6 * n ** 4}
    if kind == "inverse3d":
        return {"bytes": 16 * n ** 3, "flops": 6 * n ** 4}
    if kind == "residual3d":
        return {"bytes": 24 * n ** 3, "flops": 16 * n ** 3}
    if kind == "ex1":
        return {"bytes": 46 * 24 * n ** 3, "flops": 46 * 6 * n ** 4}
    if kind == "eig":
        return {"bytes": 650 * 16 * n ** 3, "flops": 650 * 6 * n ** 4}
    if kind == "sem":
        return {"bytes": 7 * 24 * n ** 3, "flops": 7 * (12 * n ** 4 + 6 * (case["k"] + 2) * n ** 3)}
    if kind == "batch":
        sizes = _system_sizes(case)
        pts, ops = (sum(float(m) ** p for m in sizes) / len(sizes) for p in (2, 3))
        return {"bytes": 12 * 48 * case["count"] * pts, "flops": 12 * 8 * case["count"] * ops}
    pts = case["B"] * case["G"] ** 3
    # each block: its input and pre-activation kept in 16 bits (written forward, read backward), 32 channels
    return {"bytes": pts * (4 * 4 * 64 + 8), "flops": pts * 4 * 3 * 2 * 32 * (32 + 2 * 6)}


# ---------------------------------------------------------------------------------------------
# the same results in 64 bits, with torch and numpy alone
# ---------------------------------------------------------------------------------------------
def _fd_matrix(n, h, bc):
    H = 2.0 * np.eye(n) - np.eye(n, k=1) - np.eye(n, k=-1)
    w = np.ones(n)
    if bc == "neumann":
        H[0, 1] = H[n - 1, n - 2] = -2.0
        w[0] = w[-1] = 0.5
    return H / (h * h), w


def _sem_matrix(n, k):
    xi, E, _ = _sem_nodes(n, k)
    P = np.polynomial.legendre.Legendre.basis(k)
    w = 2.0 / (k * (k + 1) * P(xi) ** 2)
    bw = np.array([1.0 / np.prod([xi[j] - xi[q] for q in range(k + 1) if q != j]) for j in range(k + 1)])
    D = np.array([[(bw[j] / bw[i]) / (xi[i] - xi[j]) if i != j else 0.0 for j in range(k + 1)] for i in range(k + 1)])
    D -= np.diag(D.sum(axis=1))
    K = 2.0 * E * (D.T * w[None, :]) @ D
    S, m = np.zeros((E * k + 1,) * 2), np.zeros(E * k + 1)
    for e in range(E):
        S[e * k:(e + 1) * k + 1, e * k:(e + 1) * k + 1] += K
        m[e * k:(e + 1) * k + 1] += w / (2.0 * E)
    S, m = S[1:-1, 1:-1], m[1:-1]
    return S / m[:, None], m


def _eig(H, w):
    """H = S diag(lam) S^-1 through the symmetric W^1/2 H W^-1/2; on the GPU."""
    r = np.sqrt(w)
    Hs = r[:, None] * H / r[None, :]
    lam, Q = np.linalg.eigh(0.5 * (Hs + Hs.T))
    return tuple(torch.from_numpy(np.ascontiguousarray(a)).to(DEV) for a in (Q / r[:, None], Q.T * r[None, :], lam))


def _mode(M, X, axis):
    n, d = X.shape[0], X.ndim
    if axis == d - 1:
        return (X.reshape(-1, n) @ M.T).reshape(X.shape)
    if axis == 0:
        return (M @ X.reshape(n, -1)).reshape(X.shape)
    return torch.matmul(M, X)


def _inverse(r, eig, shift, scale=1.0):
    S, Si, lam = eig
    d = r.ndim
    X = r
    for a in range(d):
        X = _mode(Si, X, a)
    X = X / (scale * sum(lam.reshape([-1 if a == b else 1 for b in range(d)]) for a in range(d)) + shift)
    for a in range(d):
        X = _mode(S, X, a)
    return X


def _laplacian(U, h, bc):
    out = torch.zeros_like(U)
    for a in range(U.ndim):
        W, O = torch.movedim(U, a, 0), torch.movedim(out, a, 0)
        T = 2.0 * W
        T[1:] -= W[:-1]
        T[:-1] -= W[1:]
        if bc == "neumann":
            T[0] -= W[1]
            T[-1] -= W[-2]
        O += T / (h * h)
    return out


def _newton_like(f, U, apply, eig, lam, b, V=0.0):
    """The quasi-Newton iteration, beta the mid-range of 3 b U^2 + V, to the same stop rule."""
    fn = torch.linalg.vector_norm(f)
    for _ in range(200):
        r = apply(U) + (lam + V) * U + b * U ** 3 - f
        if float(torch.linalg.vector_norm(r) / fn) <= TOL:
            break
        d = 3.0 * b * U * U + V
        U = U - _inverse(r, eig, lam + 0.5 * float(d.max() + d.min()))
    return U


def exact(case, seed):
    kind, n = case["kind"], case.get("n", 0)
    if kind in ("solve2d", "solve3d"):
        if case.get("bc") == "neumann":
            x, u, f = _ex2d1(n)
            h, U, lam, bc = 2.0 / (n - 1), u + 0.1 * _poly(x, _gen(seed), 2), 1.0, "neumann"
        else:
            f = _source(case, seed, 2 if kind == "solve2d" else 3)
            h, U, lam, bc = 1.0 / (n + 1), torch.zeros_like(f), 0.0, "dirichlet"
        U = _newton_like(f, U, lambda W: _laplacian(W, h, bc), _eig(*_fd_matrix(n, h, bc)), lam, 1.0)
        return {"U": U, "iterations": None}
    if kind == "inverse3d":
        return _inverse(_rough(n, seed), _eig(*_fd_matrix(n, 1.0 / (n + 1), "dirichlet")), 3.0)
    if kind == "residual3d":
        f, u = _source(case, seed, 3), _manufactured(n, 3, _gen(seed + 1))[0]
        R, d = _laplacian(u, 1.0 / (n + 1), "dirichlet") + u ** 3 - f, 3.0 * u * u
        lo, hi = float(d.min()), float(d.max())
        return {"R": R, "stats": [float(torch.linalg.vector_norm(R)), float(torch.linalg.vector_norm(f)), lo, hi,
                                  0.5 * (lo + hi)]}
    if kind == "ex1":
        v, f, U = _ex1(n, seed)
        h = 2.0 / (n - 1)
        U = _newton_like(f, U, lambda W: _laplacian(W, h, "neumann"), _eig(*_fd_matrix(n, h, "neumann")), 10.0, 10.0,
                         _sum3(v))
        return {"U": U, "iterations": None}
    if kind == "eig":
        v, h, U = _ex2(n, seed)
        V, eig, m = _sum3(v), _eig(*_fd_matrix(n, h, "dirichlet")), h ** 3
        U = U / torch.sqrt(m * torch.sum(U * U))
        for _ in range(4096):
            F = _laplacian(U, h, "dirichlet") + V * U + 1600.0 * U ** 3
            lm = float(m * torch.sum(F * U))
            F = F - lm * U
            if float(torch.sqrt(m * torch.sum(F * F))) <= TOL * abs(lm):
                break
            d = 4800.0 * U * U + V
            U = U - _inverse(F, eig, 0.5 * float(d.max() + d.min()) - lm)
            U = U / torch.sqrt(m * torch.sum(U * U))
        return {"U": U, "lambda": lm}
    if kind == "sem":
        f = _sem_source(case, seed)
        H, m = _sem_matrix(n, case["k"])
        Ht = torch.from_numpy(H).to(DEV)
        U = _newton_like(f, torch.zeros_like(f), lambda W: sum(_mode(Ht, W, a) for a in range(3)), _eig(H, m), 0.0, 1.0)
        return {"U": U, "iterations": None}
    if kind == "batch":
        slab, eigs = [], {}
        for m, alpha, D, f1, f2 in _systems(case, seed):
            h = 1.0 / (m + 1)
            if m not in eigs:
                eigs[m] = _eig(*_fd_matrix(m, h, "dirichlet"))
            eig = eigs[m]
            U, V = torch.zeros_like(f1), torch.zeros_like(f2)
            fn = math.sqrt(float(torch.sum(f1 * f1) + torch.sum(f2 * f2)))
            for _ in range(200):
                Fu = _laplacian(U, h, "dirichlet") + U ** 3 + alpha * V - f1
                Fv = D * _laplacian(V, h, "dirichlet") + V ** 3 - alpha * U - f2
                if math.sqrt(float(torch.sum(Fu * Fu) + torch.sum(Fv * Fv))) <= TOL * fn:
                    break
                a, d = 3.0 * U * U, 3.0 * V * V
                root = torch.sqrt(torch.clamp((a - d) ** 2 - 4.0 * alpha * alpha, min=0.0))
                beta = 0.25 * float((a + d + root).max() + (a + d - root).min())
                U, V = U - _inverse(Fu, eig, beta), V - _inverse(Fv, eig, beta, D)
            pad = torch.zeros(-(-m * m // 32) * 32 - m * m, dtype=torch.float64, device=DEV)
            slab += [U.reshape(-1), pad, V.reshape(-1), pad]
        return {"UV": torch.cat(slab), "iterations": None}
    return _net_exact(case, seed)


def _net_exact(case, seed):
    p, f, t = _net_data(case, seed)
    C, M, L, G = 32, 6, 4, case["G"]
    p = p.double().to(DEV).requires_grad_(True)
    at = [0]

    def take(*shape):
        k = math.prod(shape)
        at[0] += k
        return p[at[0] - k:at[0]].reshape(shape)

    j = torch.arange(1, G + 1, dtype=torch.float64, device=DEV)
    B = math.sqrt(2.0 / (G + 1)) * torch.sin(math.pi * j[:, None] * j[None, :M] / (G + 1))
    wl, bl = take(C), take(C)
    h = f.double().reshape(-1, G, G, G)[..., None] * wl + bl
    for layer in range(L):
        R, W, b = take(M, M, M, C, C), take(C, C), take(C)
        s = torch.einsum("bzyxc,xr->bzyrc", h, B)
        s = torch.einsum("bzyrc,yq->bzqrc", s, B)
        s = torch.einsum("bzqrc,zp->bpqrc", s, B)
        s = torch.einsum("bpqri,pqrio->bpqro", s, R)
        s = torch.einsum("bpqrc,zp->bzqrc", s, B)
        s = torch.einsum("bzqrc,yq->bzyrc", s, B)
        s = torch.einsum("bzyrc,xr->bzyxc", s, B)
        h = s + h @ W + b
        if layer < L - 1:
            h = torch.nn.functional.gelu(h, approximate="tanh")
    out = h @ take(C) + take(1)
    loss = torch.mean((out - t.double().reshape(out.shape)) ** 2)
    loss.backward()
    return {"loss": float(loss), "grads": p.grad}
