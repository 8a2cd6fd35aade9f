"""GPU: launches of the CTA-pair kernel back to back with kernels that take its SMs' shared memory over at once (the
cluster plan, whose barriers lie where a pair's late arrival would land, and the quantization).  One arrangement per entry:
one tile per pair, pairs without a second tile, a last tile with one accumulator behind tiles with two, fewer stages
than the ring holds, K cut between two pairs.  Every launch must return the bits of the first one, and no wait may run out."""
import pytest
import torch

from paper_2505_14638_b200 import binding

pytestmark = pytest.mark.gpu


def _layer(M, N, K, symmetric, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    W = torch.randn((N, K), generator=g, device="cuda") * 0.02
    tw = binding.prepack_weight(*binding.quantize_weight_rtn(W, symmetric=symmetric))
    x = torch.randn((M, K), generator=g, device="cuda").to(torch.bfloat16)
    return x, tw, binding.new_workspace(M, N, K, tw.fmt), torch.empty((M, N), dtype=torch.bfloat16, device="cuda")


@pytest.mark.parametrize("symmetric", [True, False])
@pytest.mark.parametrize("M,N,K", [(512, 6144, 1024), (700, 12304, 640), (1152, 9488, 384), (4700, 9488, 256), (9000, 9488, 128),
                                   (511, 2048, 8192)])
def test_launches_back_to_back(M, N, K, symmetric):
    x, tw, ws, y = _layer(M, N, K, symmetric, M + N + K)
    xc, twc, wsc, yc = _layer(40, 4096, 1024, symmetric, 3)
    xq, sq = binding.quantize_act(x)
    xcq, scq = binding.quantize_act(xc)
    want = binding.linear_tiled(xq, sq, tw, workspace=ws).clone()
    wantc = binding.linear_tiled(xcq, scq, twc, workspace=wsc).clone()
    for _ in range(8):
        for _ in range(4):
            binding.linear_tiled(xq, sq, tw, out=y, workspace=ws)
            binding.linear_tiled(xcq, scq, twc, out=yc, workspace=wsc)
        binding.quantize_act(x, out=(xq, sq))
        binding.linear_tiled(xq, sq, tw, out=y, workspace=ws)
        assert torch.equal(y, want) and torch.equal(yc, wantc)
    assert binding.query_device_status() == 0
