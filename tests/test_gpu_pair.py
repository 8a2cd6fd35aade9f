"""GPU: the CTA-pair kernel (more than 128 tokens) at the edges of its tiles and of its three arrangements: ragged last
channel tiles (one of the pair's CTAs with few rows or none), ragged token tiles on both sides of an accumulator of
256 tokens, K of one k-block (stages that run several tiles ahead) to many, K cut unevenly between two pairs, several
tiles per pair, FP32 outputs, and a pitch of Y that no 16-byte store fits.

Tolerance: a float64 product of the same FP8 operands is exact; the tensor core's FP32 sums of K terms are within
K 2^-24 of the sum of magnitudes, which for these random signs is below 4 sqrt(K) times the result's scale."""
import numpy as np
import pytest
import torch

from gpu_utils import Guarded, bf16_dev
from paper_2505_14638_b200 import binding, inputs

pytestmark = pytest.mark.gpu

SHAPES = [
    # 256 x 256 tiles: one tile per pair; two rounds, 147 tiles on 74 pairs; and (sign-magnitude) 256 x 512 with one accumulator
    (129, 28672, 1280), (512, 6144, 4096), (700, 12304, 2048),
    # 256 x 512 tiles: last token tile of at most 256 tokens, of more, of one token; several rounds; K = 128 and 256
    (1030, 16400, 1024), (2100, 9232, 640), (4609, 9488, 384), (513, 18448, 1152), (9000, 9488, 128), (4700, 9488, 256),
    # K cut between two pairs: 64 and 65 k-blocks, a second CTA with 16 rows, with none
    (511, 2048, 8192), (300, 2064, 8320), (257, 2192, 14336),
]


@pytest.mark.parametrize("asym", [False, True])
@pytest.mark.parametrize("M,N,K", SHAPES)
def test_edges_of_tiles_and_arrangements(M, N, K, asym):
    dev = torch.device("cuda")
    W = torch.from_numpy(inputs.make_weight(N, K, 0.02, seed=M + N)).to(dev)
    codes, gs, gz, sw = binding.quantize_weight_rtn(W, symmetric=not asym, per_channel=asym)
    del W
    w8 = binding.dequant_weight(codes, gs, gz).view(torch.float8_e4m3fn)
    tw = binding.prepack_weight(codes, gs, gz, sw)
    x8, s_x = binding.quantize_act(bf16_dev(inputs.make_activation(M, K, M + K, 0.01, 20.0)))
    rng = np.random.default_rng(N)
    cols = torch.from_numpy(np.unique(np.concatenate([rng.choice(N, 96, replace=False), np.arange(16), np.arange(N - 144, N)]))).to(dev)
    scale = (sw[cols] if sw.numel() > 1 else sw).double()
    ref = (x8.view(torch.float8_e4m3fn).double() @ w8[cols].double().t()) * s_x.double()[:, None] * scale[None, :]
    mag = (x8.view(torch.float8_e4m3fn).double().square() @ w8[cols].double().square().t()).sqrt() * s_x.double()[:, None] * scale[None, :]
    ws = binding.new_workspace(M, N, K, tw.fmt, dev)
    y32 = Guarded((M, N), torch.float32, 777.0)
    binding.linear_tiled(x8, s_x, tw, out_dtype=binding.OUT_FP32, out=y32.t, workspace=ws)
    y32.check()
    assert binding.query_device_status() == 0
    bound = 4.0 * K ** 0.5 * 2.0 ** -24 * K ** 0.5 * mag + 1e-30
    assert bool(((y32.t[:, cols].double() - ref).abs() <= bound).all())
    assert not bool((y32.t == 777.0).any())
    for pitch in (N, N + 8, N + 4):   # 16-byte stores with and without a gap behind a row; and none
        y = Guarded((M, pitch), torch.bfloat16, 777.0)
        for _ in range(2):
            binding.linear_tiled(x8, s_x, tw, out=y.t[:, :N], workspace=ws)
        y.check()
        assert torch.equal(y.t[:, :N], y32.t.to(torch.bfloat16))   # the same sums, rounded once
        assert bool((y.t[:, N:] == 777.0).all())
    assert binding.query_device_status() == 0
    assert not bool(ws.any())   # needs no workspace
