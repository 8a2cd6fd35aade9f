"""GPU: prepacked groups with a zero-point, expanded as pairs of one sign: every zero-point (also ones past 15, which make all
values negative) with scales of both signs, subnormal, at and past the value from which everything saturates.

The activations are rows of the identity, so an output is one expanded weight: exact, no tolerance (zeros of either sign)."""
import numpy as np
import pytest
import torch

from gpu_utils import bf16_dev, dev
from paper_2505_14638_b200 import binding

pytestmark = pytest.mark.gpu

SCALES = [0x3F80, 0xBF80, 0x41C8, 0xC1C8, 0x3B03, 0x0001, 0x8001, 0x0000, 0x43DF, 0x43E0, 0x43E1, 0xC3E1, 0x7F7F, 0xFF7F, 0x3A80, 0x4085]


def _weights(N, K, seed):
    rng = np.random.default_rng(seed)
    codes = rng.integers(0, 256, (N, K // 2), dtype=np.uint8)
    g = np.arange(N * (K // 128)).reshape(N, K // 128)
    gzero = (g % 17).astype(np.uint8)
    gzero[gzero == 16] = 255
    gscale = np.array(SCALES, dtype=np.uint16)[(g // 17) % len(SCALES)]
    return dev(codes), bf16_dev(gscale), dev(gzero)


@pytest.mark.parametrize("M,N,K", [(1, 1024, 256), (16, 1024, 384), (8, 19216, 256), (64, 1040, 256), (100, 19216, 128),
                                   (256, 1040, 256), (640, 9616, 640),
                                   # weights to registers: also an odd number of units per CTA, k-blocks that are no multiple of four
                                   (8, 2048, 896), (16, 1024, 2048), (5, 2384, 640), (16, 1216, 1792)])
@pytest.mark.parametrize("chain", [False, True])
def test_every_zero_point_expands_to_the_dequantized_weights(M, N, K, chain):
    if chain and M > 16:
        pytest.skip("a chain problem has at most 16 tokens")
    codes, gs, gz = _weights(N, K, M + N)
    one = torch.ones(1, device="cuda")
    w = binding.dequant_weight(codes, gs, gz).view(torch.float8_e4m3fn).float()
    tw = binding.prepack_weight(codes, gs, gz, one)
    assert tw.fmt == binding.FMT_TILED
    cols = torch.arange(M, device="cuda") * (K - 1) // max(M - 1, 1)    # first to last column
    x = torch.zeros((M, K), dtype=torch.bfloat16, device="cuda")
    x[torch.arange(M, device="cuda"), cols] = 1.0
    y = torch.full((M, N), 777.0, device="cuda")
    if chain:
        unit = torch.ones(1, device="cuda")
        binding.LinearChain([dict(x=x, weight=tw, y=y, static_scale=unit)])()
    else:
        x8, s_x = binding.quantize_act(x, static_scale=torch.ones(1, device="cuda"))
        binding.linear_tiled(x8, s_x, tw, out_dtype=binding.OUT_FP32, out=y)
    assert binding.query_device_status() == 0
    assert torch.equal(y, w[:, cols].t())


def test_a_buffer_of_integer_zero_points_reads_as_nan():
    N, K = 1024, 256
    codes, gs, gz = _weights(N, K, 3)
    one = torch.ones(1, device="cuda")
    tw = binding.prepack_weight(codes, gs, gz, one)
    meta = tw.buf[N * K // 2:].view(torch.int32)
    meta.copy_(torch.arange(meta.numel(), device="cuda", dtype=torch.int32) % 16 << 16 | 0x3F80)
    x8, s_x = binding.quantize_act(torch.ones((4, K), dtype=torch.bfloat16, device="cuda"))
    assert bool(binding.linear_tiled(x8, s_x, tw).isnan().all())


@pytest.mark.parametrize("M,N,K", [(4, 2048, 896), (16, 1024, 384), (64, 1040, 256), (256, 1040, 256)])
def test_scales_that_are_not_finite(M, N, K):
    # 0 x infinity is NaN, so an infinite scale gives NaN for the codes at the zero-point and +-448 for the others; one such
    # weight, or a NaN scale, makes the row's outputs NaN.  Every other row has no code at the zero-point.
    codes, gs, gz = _weights(N, K, 5)
    u = torch.stack((codes & 15, codes >> 4), -1).reshape(N, K // 128, 128).int()
    z = gz.int()[:, :, None]
    u[::2] = torch.where(u[::2] == z[::2], (u[::2] + 1) % 16, u[::2])
    u = u.reshape(N, K // 2, 2)
    codes = (u[:, :, 0] | u[:, :, 1] << 4).to(torch.uint8).contiguous()
    odd = bf16_dev(np.array([0x7F80, 0xFF80, 0x7F80, 0xFF80, 0x7FC0, 0xFFFF], dtype=np.uint16))
    gs[:, K // 128 - 1] = odd[torch.arange(N, device="cuda") // 2 % 6]
    one = torch.ones(1, device="cuda")
    w = binding.dequant_weight(codes, gs, gz).view(torch.float8_e4m3fn).double()
    x = torch.zeros((M, K), dtype=torch.bfloat16, device="cuda")
    x[torch.arange(M, device="cuda"), torch.arange(M, device="cuda") * (K - 1) // (M - 1)] = 1.0
    x8, s_x = binding.quantize_act(x, static_scale=one)
    want = x.double() @ w.t()
    assert bool(want.isnan().any()) and bool((want.abs() == 448).any())
    y = binding.linear_tiled(x8, s_x, binding.prepack_weight(codes, gs, gz, one), out_dtype=binding.OUT_FP32).double()
    assert binding.query_device_status() == 0
    assert torch.equal(y.isnan(), want.isnan()) and torch.equal(y.nan_to_num(), want.nan_to_num())
