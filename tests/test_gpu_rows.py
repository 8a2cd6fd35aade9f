"""GPU: up to 128 tokens on layers whose rows are dealt out to the SMs in contiguous runs (linear_rows_kernel): one and two blocks
of 128 rows per run, more runs than SMs, an odd number of k-blocks, K cut through the workspace, CTAs of half an SM, rows of Y that
16-byte stores do not fit.

Tolerance: FP32 sums of K exact products against float64, 4 K 2^-24 of the root of the summed squares."""
import numpy as np
import pytest
import torch

from gpu_utils import Guarded, bf16_dev
from paper_2505_14638_b200 import binding, inputs

pytestmark = pytest.mark.gpu

# What w4a8_linear takes linear_rows_kernel for on 148 SMs (test_decode_plan.py holds decode_choice to it): CTAs of whole SMs,
ROWS = [
    (1, 18944, 2176), (16, 18960, 2304), (8, 37888, 1792), (3, 37904, 1920),      # 128 / 136 / 256 rows a run, two runs a CTA
    (17, 9488, 4224), (64, 19216, 2176), (65, 18944, 3200), (128, 28688, 2176), (100, 37904, 2304),
    (128, 18944, 3200),                                    # with zero-points as many stages as groups in both rings
    (16, 1552, 14336), (13, 1024, 8320), (1, 4096, 5760), (12, 9472, 3456), (9, 1024, 8320), (14, 128, 4096), (16, 16, 4224)]   # K cut
# ... with zero-points whole tiles take their place (few tiles, K not cut),
ROWS_SIGNMAG = [(128, 7664, 3072), (44, 6384, 1792)]
# and CTAs of half an SM, the first four with K cut.
ROWS_HALF = [(9, 1008, 5888), (12, 4400, 3200), (2, 128, 4096), (4, 16, 4224), (1, 9488, 640), (16, 18960, 1408), (5, 37904, 896),
             (8, 37888, 1664)]


def _layer(M, N, K, asym):
    W = torch.from_numpy(inputs.make_weight(N, K, 0.02, seed=M + N + K)).cuda()
    codes, gs, gz, sw = binding.quantize_weight_rtn(W, symmetric=not asym, per_channel=asym)
    w64 = binding.dequant_weight(codes, gs, gz).view(torch.float8_e4m3fn).double()
    x8, s_x = binding.quantize_act(bf16_dev(inputs.make_activation(M, K, M + K, 0.01, 20.0)))
    x64 = x8.view(torch.float8_e4m3fn).double()
    scale = s_x.double()[:, None] * (sw.double() if sw.numel() > 1 else sw.double().reshape(1))[None, :]
    ref, mag = (x64 @ w64.t()) * scale, (x64.square() @ w64.square().t()).sqrt() * scale
    return x8, s_x, binding.prepack_weight(codes, gs, gz, sw), ref, mag


@pytest.mark.parametrize("asym", [False, True])
@pytest.mark.parametrize("M,N,K", ROWS + ROWS_SIGNMAG + ROWS_HALF)
def test_rows_in_runs(M, N, K, asym):
    x8, s_x, tw, ref, mag = _layer(M, N, K, asym)
    ws = binding.new_workspace(M, N, K, tw.fmt, "cuda")
    outs = []
    for rep in range(2):
        y = Guarded((M, N), torch.float32, 777.0)
        binding.linear_tiled(x8, s_x, tw, out_dtype=binding.OUT_FP32, out=y.t, workspace=ws)
        y.check()
        outs.append(y.t)
        assert not bool(ws[:65536].any())          # counters left at zero
    assert binding.query_device_status() == 0
    assert bool(((outs[0].double() - ref).abs() <= 4.0 * K * 2.0 ** -24 * mag + 1e-30).all())
    assert torch.equal(outs[0], outs[1])
    yb = binding.linear_tiled(x8, s_x, tw, workspace=ws)
    assert torch.equal(yb, outs[0].to(torch.bfloat16))


@pytest.mark.parametrize("M,N,K", [(5, 18944, 2176), (40, 28688, 2304), (16, 1552, 14336), (7, 18960, 896)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_rows_of_y_that_wide_stores_do_not_fit(M, N, K, dtype):
    x8, s_x, tw, ref, _ = _layer(M, N, K, True)
    ws = binding.new_workspace(M, N, K, tw.fmt, "cuda")
    out_dtype = binding.OUT_FP32 if dtype == torch.float32 else binding.OUT_BF16
    want = binding.linear_tiled(x8, s_x, tw, out_dtype=out_dtype, workspace=ws)
    wide = Guarded((M, N + 3), dtype, 7.0)
    binding.linear_tiled(x8, s_x, tw, out_dtype=out_dtype, out=wide.t[:, :N], workspace=ws)
    wide.check()
    assert torch.equal(wide.t[:, :N], want) and bool((wide.t[:, N:] == 7.0).all())


@pytest.mark.parametrize("asym", [False, True])
@pytest.mark.parametrize("M,N,K", [(4, 1552, 8320), (16, 4096, 4096), (3, 18960, 2176)])
def test_without_a_workspace_k_is_not_cut(M, N, K, asym):
    # The bits of one chain of sums over K: of a chain launch on the layer's rows, repeated until every SM has a whole block of 96 of
    # them, whose K it does not cut.
    W = torch.from_numpy(inputs.make_weight(N, K, 0.02, seed=M + N + K)).cuda()
    q = binding.quantize_weight_rtn(W, symmetric=not asym, per_channel=False)
    x = bf16_dev(inputs.make_activation(M, K, M + K, 0.01, 20.0))
    x8, s_x = binding.quantize_act(x)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    whole = 96 * sms
    rows = torch.arange(max(whole, N) // 16 * 16, device="cuda") % N
    many = binding.prepack_weight(*[None if t is None else t[rows].contiguous() for t in q[:3]], q[3])
    chain = torch.zeros((M, rows.numel()), dtype=torch.float32, device="cuda")
    binding.LinearChain([dict(x=x, weight=many, y=chain)])()
    tiny = torch.zeros(16, dtype=torch.uint8, device="cuda")
    y = binding.linear_tiled(x8, s_x, binding.prepack_weight(*q), out_dtype=binding.OUT_FP32, workspace=tiny)
    assert binding.query_device_status() == 0
    n = min(N, whole)
    assert torch.equal(y[:, :n], chain[:, :n])
