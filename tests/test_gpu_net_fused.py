"""The fused training kernels of the warm-start network against the FP64 oracle: odd grids, every
rounding of the mode count, one block (first and last at once), one sample and many."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


# rows of 16 nodes and items of 16 rows with remainders; odd mode counts are padded to even; the
# last case (nine modes) keeps the unfused kernels
@pytest.mark.parametrize("G,M,L,B", [(9, 2, 1, 1), (16, 3, 2, 2), (17, 4, 1, 3), (23, 5, 2, 1), (31, 6, 3, 2),
                                     (33, 7, 1, 9), (24, 8, 2, 1), (12, 9, 2, 2), (8, 6, 16, 1)])
def test_loss_gradients_and_output(G, M, L, B):
    import torch

    from oracle import no_oracle as O
    from paper_2502_03611_gb300 import qn
    rng = np.random.default_rng(100 * G + M)
    net = qn.QnNet(G, M, L, max_batch=B + 1)
    p = rng.standard_normal(net.nparams) * 0.15
    p = p.astype(np.float32)
    net.set_params(p)
    f = rng.standard_normal((B, G, G, G)).astype(np.float32)
    tgt = rng.standard_normal((B, G, G, G)).astype(np.float32)
    ft, tt = torch.from_numpy(f).cuda().reshape(-1), torch.from_numpy(tgt).cuda().reshape(-1)
    grads = torch.empty(net.nparams, dtype=torch.float32, device="cuda")
    loss = net.gradients(ft, tt, B, grads)
    out = torch.empty_like(ft)
    net.forward(ft, out, B)
    lo, oo, go = O.loss_and_grads(p, f.astype(np.float64), tgt.astype(np.float64), 32, M, L)
    # BF16 activations (2^-9 each) through L blocks; sums over many nodes average them
    tol = 2.0 ** -9 * (2 + 2 * L)
    assert abs(loss - lo) <= tol * abs(lo)
    assert np.linalg.norm(out.cpu().numpy() - oo.ravel()) <= tol * np.linalg.norm(oo)
    g = grads.cpu().numpy().astype(np.float64)
    assert np.linalg.norm(g - go) <= tol * np.linalg.norm(go)
    # every parameter group on its own (a wrong small group hides in the whole norm)
    at = 0
    sizes = [32, 32] + [M ** 3 * 1024, 1024, 32] * L + [32, 1]
    for n in sizes:
        a, b = g[at:at + n], go[at:at + n]
        assert np.linalg.norm(a - b) <= 4 * tol * np.linalg.norm(b) + 1e-7 * np.linalg.norm(go), (at, n)
        at += n
