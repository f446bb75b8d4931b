"""Device memory of a network: with 2 to 8 modes only what the fused kernels use.

Per node and sample: 64 bytes for each block's input, 64 for each block's z but the last's, 128 for
the gradient, 8 for output and its gradient; the mode sums and parameters of these sizes are
below 24 MB, and each of the 30 or so allocations is rounded up to at most 2 MB.
"""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("G,M,L,B", [(64, 6, 2, 8), (48, 4, 3, 16)])
def test_memory_of_a_fused_network(G, M, L, B):
    import torch

    from paper_2502_03611_gb300 import qn
    qn.load_library()
    qn.QnNet(8, 2, 1, max_batch=1)   # the kernels' code is loaded
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    net = qn.QnNet(G, M, L, max_batch=B)
    used = free - torch.cuda.mem_get_info()[0]
    assert used <= B * G ** 3 * (64 * L + 64 * (L - 1) + 128 + 8) + (24 << 20) + 30 * (2 << 20)
    f = torch.randn(B * G ** 3, device="cuda")
    grads = torch.empty(net.nparams, dtype=torch.float32, device="cuda")
    assert net.gradients(f, f, B, grads) >= 0.0
