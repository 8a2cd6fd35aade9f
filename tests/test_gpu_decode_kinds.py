"""GPU: up to 128 tokens on prepacked layers, shapes on both sides of the limits between the kernels (decode_shapes.py, which
test_decode_plan.py holds to the kernels they stand for).

Tolerance: FP32 sums of K exact products against float64, 4 K 2^-24 of the root of the summed squares."""
import pytest
import torch

from decode_shapes import SHAPES
from gpu_utils import Guarded
from paper_2505_14638_b200 import binding
from test_gpu_rows import _layer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,M,N,K,symmetric", [(k, *s) for k in sorted(SHAPES) for s in SHAPES[k]])
def test_both_sides_of_the_limits_between_kernels(kind, M, N, K, symmetric):
    x8, s_x, tw, ref, mag = _layer(M, N, K, not symmetric)
    ws = binding.new_workspace(M, N, K, tw.fmt, "cuda")
    outs = []
    for rep in range(2):
        y = Guarded((M, N), torch.float32, 777.0)
        binding.linear_tiled(x8, s_x, tw, out_dtype=binding.OUT_FP32, out=y.t, workspace=ws)
        y.check()
        outs.append(y.t)
    assert binding.query_device_status() == 0
    assert not bool(ws[:65536].any())          # control data left at zero, or never touched
    assert bool(((outs[0].double() - ref).abs() <= 4.0 * K * 2.0 ** -24 * mag + 1e-30).all())
    assert torch.equal(outs[0], outs[1])
    yb = binding.linear_tiled(x8, s_x, tw, workspace=ws)
    assert torch.equal(yb, outs[0].to(torch.bfloat16))


@pytest.mark.parametrize("M,N,K,asym", [(8, 4096, 3840, False), (3, 4128, 4864, True), (12, 1008, 5760, False), (1, 5248, 3200, True)])
def test_launches_that_share_sms_share_a_workspace_in_turn(M, N, K, asym):
    # CTAs of half an SM, K cut: a launch starts beside the one before and uses the same counters and partial sums
    x8, s_x, tw, ref, mag = _layer(M, N, K, asym)
    other = [_layer(M, N, K + 128 * i, asym) for i in (1, 2)]
    ws = binding.new_workspace(M, N, K, tw.fmt, "cuda")
    runs = [(x8, s_x, tw)] + [o[:3] for o in other]
    want = [binding.linear_tiled(*r, out_dtype=binding.OUT_FP32, workspace=ws) for r in runs]
    ys = [torch.zeros((M, N), device="cuda") for _ in range(60)]
    for i, y in enumerate(ys):
        binding.linear_tiled(*runs[i % 3], out_dtype=binding.OUT_FP32, out=y, workspace=ws)
    torch.cuda.synchronize()
    assert binding.query_device_status() == 0 and not bool(ws[:65536].any())
    assert all(torch.equal(y, want[i % 3]) for i, y in enumerate(ys))
    assert bool(((want[0].double() - ref).abs() <= 4.0 * K * 2.0 ** -24 * mag + 1e-30).all())
