"""GPU: the quantizer on a layer large enough that its steps apply the errors of two blocks at a time, and change over to one
block at a time on the way.  Rows do not depend on one another (per-channel scales), so slabs of the same rows, quantized on
their own with one block at a time (the route that test_gpu_dpq.py compares with the oracle), must give the same bits.
Odd and even numbers of blocks; a last row tile that is not full."""
import pytest
import torch

from paper_2505_14638_b200 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K,symmetric", [(4112, 5248, False), (8208, 3072, True), (8192, 2944, False)])
def test_large_layers_in_slabs(N, K, symmetric):
    g = torch.Generator(device="cuda")
    g.manual_seed(N + K)
    W = torch.randn((N, K), generator=g, device="cuda") * 0.02
    U = (torch.eye(K, device="cuda") + 0.5 * torch.triu(torch.randn((K, K), generator=g, device="cuda"), 1) / K ** 0.5).contiguous()
    whole = binding.dpq_quantize(W, U, None, symmetric=symmetric, mse_steps=3, per_channel=True)
    for r0 in list(range(0, 1024, 256)) + [N - 272]:
        slab = binding.dpq_quantize(W[r0:r0 + 272].contiguous(), U, None, symmetric=symmetric, mse_steps=3, per_channel=True)
        for a, b in zip(whole, slab):
            if a is not None:
                assert torch.equal(a[r0:r0 + 272].view(torch.uint8), b.view(torch.uint8))
