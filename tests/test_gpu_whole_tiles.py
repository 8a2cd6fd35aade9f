"""GPU: 17..128 tokens on layers with more tiles of 128 channels than the cluster plan takes: whole tiles of the persistent
kernel, which need no workspace, and linear_rows_kernel for a longer K.
Edges: 17, 64, 65 and 128 tokens, a ragged last tile, one more tile than SMs, one k-block (the rule's limits: decode_shapes.py).

Tolerance as in test_gpu_pair.py: FP32 sums of K exact products against float64."""
import numpy as np
import pytest
import torch

from gpu_utils import Guarded, bf16_dev
from paper_2505_14638_b200 import binding, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("asym", [False, True])
@pytest.mark.parametrize("M,N,K", [(17, 9616, 128), (64, 9616, 1408), (65, 9616, 1408), (128, 18944, 256), (33, 18960, 2944),
                                   (32, 18960, 3072), (77, 19216, 6016), (100, 19216, 6144), (128, 28672, 1024)])
def test_wide_layers_of_17_to_128_tokens(M, N, K, asym):
    dev = torch.device("cuda")
    W = torch.from_numpy(inputs.make_weight(N, K, 0.02, seed=M + N)).to(dev)
    codes, gs, gz, sw = binding.quantize_weight_rtn(W, symmetric=not asym, per_channel=asym)
    del W
    w8 = binding.dequant_weight(codes, gs, gz).view(torch.float8_e4m3fn)
    tw = binding.prepack_weight(codes, gs, gz, sw)
    x8, s_x = binding.quantize_act(bf16_dev(inputs.make_activation(M, K, M + K, 0.01, 20.0)))
    x64, w64 = x8.view(torch.float8_e4m3fn).double(), w8.double()
    scale = s_x.double()[:, None] * (sw.double() if sw.numel() > 1 else sw.double().reshape(1))[None, :]
    ref, mag = (x64 @ w64.t()) * scale, (x64.square() @ w64.square().t()).sqrt() * scale
    outs = []
    for ws in (None, binding.new_workspace(M, N, K, tw.fmt, dev)):
        y = Guarded((M, N), torch.float32, 777.0)
        binding.linear_tiled(x8, s_x, tw, out_dtype=binding.OUT_FP32, out=y.t, workspace=ws)
        y.check()
        outs.append(y.t)
        assert ws is None or not bool(ws[:65536].any())   # (control data left zero-filled, or never touched)
    assert binding.query_device_status() == 0
    assert bool(((outs[0].double() - ref).abs() <= 4.0 * K * 2.0 ** -24 * mag + 1e-30).all())
    assert torch.equal(outs[0], outs[1])
    yb = binding.linear_tiled(x8, s_x, tw, workspace=None)
    assert torch.equal(yb, outs[0].to(torch.bfloat16))
