"""Precision of the fused training kernels: they keep FP32 operands as three BF16 levels, round to
BF16 only where an activation is stored, and form gelu and its derivative in FP32.

The reference is the FP64 oracle with its activations rounded to BF16 at the same places. One block
whose input is exact in BF16 (small multiples of 1/8) leaves FP32 arithmetic alone in the
gradients of W, R and the lift: sums of up to a few hundred terms per thread and block, 2^-24
each, so 1e-6 of a group's norm. A lost third level of W or dz is 2^-18 of an operand: the CPU
test plants it in the oracle and checks that it breaks the bound. Two blocks put one gelu in
between, whose BF16 roundings (2^-9 where an FP32 error crosses a rounding point, at most 1e-4 of
the values) leave 2^-9 sqrt(1e-4) = 2e-5 in the gradients behind it, 1e-4 allowed with the second
block's.
"""
import numpy as np
import pytest

from oracle import no_oracle as O

C = 32


def _bf16(x):
    """Rounded to BF16 (to nearest even), in FP64."""
    b = np.asarray(x, np.float32).view(np.uint32)
    b = (b + 0x7FFF + ((b >> 16) & 1)) & np.uint32(0xFFFF0000)
    return b.view(np.float32).astype(np.float64)


def _levels(x, count):
    """The sum of the first `count` BF16 levels of x."""
    out = np.zeros_like(x)
    for _ in range(count):
        out = out + _bf16(x - out)
    return out


def _round_f32(x):
    return np.asarray(x, np.float32).astype(np.float64)


def _case(G, M, L, B, seed):
    rng = np.random.default_rng(seed)
    f = rng.integers(-8, 9, size=(B, G, G, G)) / 4.0
    wl, bl = rng.choice([-1.0, -0.5, 0.5, 1.0], C), rng.integers(-8, 9, C) / 8.0
    parts = [wl, bl]
    for _ in range(L):
        parts += [rng.standard_normal(M ** 3 * C * C) * 0.2, rng.standard_normal(C * C) * 0.18, rng.standard_normal(C) * 0.1]
    parts += [rng.standard_normal(C), [0.0]]
    p = np.concatenate(parts).astype(np.float32)
    # targets far above the output: the output's own rounding does not show in the gradients
    tgt = (rng.standard_normal((B, G, G, G)) * 1000.0).astype(np.float32)
    return p, f, tgt


def _oracle(p, f, tgt, M, L, wl_w=3, wl_dz=3):
    """Loss gradients and output with stored activations in BF16; W and dz of the 32 x 32 products cut
    to wl_w and wl_dz levels."""
    P = O.unpack(p, C, M, L)
    G = f.shape[1]
    Bm = _round_f32(O.sine_analysis_basis(G, M))
    h, hs, zs, hhs = _bf16(f[..., None] * P["wl"] + P["bl"]), [], [], []
    for l, (R, W, b) in enumerate(P["blocks"]):
        hh = O._analysis(h, Bm)
        z = O._synthesis(np.einsum("bpqri,pqrio->bpqro", hh, R), Bm) + h @ _levels(W, wl_w) + b
        hs.append(h)
        hhs.append(hh)
        zs.append(_bf16(z))
        h = _bf16(z) if l == L - 1 else _bf16(O.gelu(z))
    out = h @ P["wp"] + P["bp"][0]
    dout = 2.0 * (out - tgt) / out.size
    grads = {"wp": np.einsum("bzyxc,bzyx->c", h, dout), "bp": np.array([dout.sum()])}
    dh = dout[..., None] * P["wp"]
    for l in reversed(range(L)):
        R, W, b = P["blocks"][l]
        dz = dh if l == L - 1 else dh * O.gelu_grad(zs[l])
        dg = O._analysis(dz, Bm)
        cut = _levels(dz, wl_dz)
        grads[f"W{l}"] = np.einsum("bzyxi,bzyxo->io", hs[l], cut)
        grads[f"b{l}"] = dz.sum(axis=(0, 1, 2, 3))
        grads[f"R{l}"] = np.einsum("bpqri,bpqro->pqrio", hhs[l], dg)
        dh = O._synthesis(np.einsum("bpqro,pqrio->bpqri", dg, R), Bm) + cut @ _levels(W, wl_w).T
    grads["wl"], grads["bl"] = np.einsum("bzyx,bzyxc->c", f, dh), dh.sum(axis=(0, 1, 2, 3))
    return out, grads


def _groups(flat, M, L):
    P = O.unpack(flat, C, M, L)
    g = {"wl": P["wl"], "bl": P["bl"], "wp": P["wp"], "bp": P["bp"]}
    for l, (R, W, b) in enumerate(P["blocks"]):
        g[f"R{l}"], g[f"W{l}"], g[f"b{l}"] = R, W, b
    return g


def _rel(a, b):
    return np.linalg.norm(np.ravel(a) - np.ravel(b)) / np.linalg.norm(np.ravel(b))


FP32_TOL, BF16_TOL = 1e-6, 1e-4
ONE_BLOCK = [(33, 3, 1, 2), (17, 6, 1, 3), (40, 8, 1, 1)]


@pytest.mark.parametrize("case", ONE_BLOCK)
def test_a_lost_level_would_show(case):
    G, M, L, B = case
    p, f, tgt = _case(G, M, L, B, 5)
    _, want = _oracle(p, f, tgt, M, L)
    _, lost = _oracle(p, f, tgt, M, L, wl_dz=2)
    assert _rel(lost["W0"], want["W0"]) > FP32_TOL
    _, lost = _oracle(p, f, tgt, M, L, wl_w=2)
    assert max(_rel(lost["wl"], want["wl"]), _rel(lost["bl"], want["bl"])) > FP32_TOL
    # of the forward product, the second level: the third is below the output's own BF16 rounding
    assert _rel(_oracle(p, f, tgt, M, L, wl_w=1)[0], _oracle(p, f, tgt, M, L)[0]) > BF16_TOL


@pytest.fixture(scope="module")
def qn():
    from paper_2502_03611_gb300 import qn as q
    q.load_library()
    return q


def _run(qn, p, f, tgt, G, M, L, B):
    import torch
    net = qn.QnNet(G, M, L, max_batch=B)
    net.set_params(p)
    ft, tt = (torch.from_numpy(np.ascontiguousarray(a, np.float32)).cuda().reshape(-1) for a in (f, tgt))
    grads = torch.empty(net.nparams, dtype=torch.float32, device="cuda")
    net.gradients(ft, tt, B, grads)
    out = torch.empty_like(ft)
    net.forward(ft, out, B)
    return out.cpu().numpy().reshape(f.shape), _groups(grads.cpu().numpy().astype(np.float64), M, L)


@pytest.mark.gpu
@pytest.mark.parametrize("case", ONE_BLOCK)
def test_one_block_in_fp32(qn, case):
    G, M, L, B = case
    p, f, tgt = _case(G, M, L, B, 5)
    _, want = _oracle(p, f, tgt, M, L)
    _, got = _run(qn, p, f, tgt, *case)
    # (b and bp are multiples of the one sum of dout, which cancels to any size and passes no product)
    for k in ("wl", "bl", "R0", "W0"):
        assert _rel(got[k], want[k]) <= FP32_TOL, k
    assert _rel(got["wp"], want["wp"]) <= BF16_TOL


@pytest.mark.gpu
@pytest.mark.parametrize("case", [(24, 4, 2, 2), (17, 7, 2, 1)])
def test_two_blocks(qn, case):
    G, M, L, B = case
    p, f, tgt = _case(G, M, L, B, 7)
    out, want = _oracle(p, f, tgt, M, L)
    got_out, got = _run(qn, p, f, tgt, *case)
    assert _rel(got_out, out) <= BF16_TOL
    for k in set(want) - {"bp", "b1"}:
        assert _rel(got[k], want[k]) <= BF16_TOL, k
