"""GPU: every arrangement that w4a8_linear has for more than 128 tokens on prepacked weights, at the shapes of prefill_shapes.py.
Launches on fresh zero-filled workspaces agree bit for bit and are right (a repeat on a used workspace cannot show a partial
sum that is read too early); guard bands around Y and a workspace of exactly the size that is asked for stay
untouched; the workspace's control area is left zero-filled; its data is written where K is cut between CTAs and nowhere
else, which shows that the shape takes the arrangement it stands for.

Tolerance as in test_gpu_pair.py: FP32 sums of K exact products against float64 products of the same FP8 operands."""
import pytest
import torch

from gpu_utils import Guarded, bf16_dev
from paper_2505_14638_b200 import binding, inputs
from prefill_shapes import SHAPES

pytestmark = pytest.mark.gpu

CTL = 65536   # bytes of control data at the start of a workspace


def _layer(M, N, K, symmetric):
    W = torch.from_numpy(inputs.make_weight(N, K, 0.02, seed=M + N)).cuda()
    codes, gs, gz, sw = binding.quantize_weight_rtn(W, symmetric=symmetric, per_channel=not symmetric)
    del W
    x8, s_x = binding.quantize_act(bf16_dev(inputs.make_activation(M, K, M + K, 0.01, 20.0)))
    return codes, gs, gz, sw, x8, s_x, binding.prepack_weight(codes, gs, gz, sw)


@pytest.mark.parametrize("kind,M,N,K,symmetric", [(k, *s) for k, v in SHAPES.items() for s in v])
def test_fresh_launches_agree_and_are_right(kind, M, N, K, symmetric):
    codes, gs, gz, sw, x8, s_x, tw = _layer(M, N, K, symmetric)
    w64 = binding.dequant_weight(codes, gs, gz).view(torch.float8_e4m3fn).double()
    x64 = x8.view(torch.float8_e4m3fn).double()
    scale = s_x.double()[:, None] * sw.double().reshape(1, -1)
    ref, mag = (x64 @ w64.t()) * scale, (x64.square() @ w64.square().t()).sqrt() * scale
    need = binding.linear_workspace_bytes(M, N, K, weight_format=tw.fmt)
    first = None
    for pitch, dtype, out in ((N, torch.float32, binding.OUT_FP32), (N + 8, torch.float32, binding.OUT_FP32),
                              (N + 4, torch.bfloat16, binding.OUT_BF16)):
        ws = Guarded((need,), torch.uint8, 0)
        y = Guarded((M, pitch), dtype, 777.0)
        binding.linear_tiled(x8, s_x, tw, out_dtype=out, out=y.t[:, :N], workspace=ws.t)
        y.check()
        ws.check()
        assert binding.query_device_status() == 0
        assert bool((y.t[:, N:] == 777.0).all())
        assert not bool(ws.t[:CTL].any())
        assert bool(ws.t[CTL:].any()) == kind.startswith("cut")
        if first is None:
            first = y.t
            assert bool(((first.double() - ref).abs() <= 4.0 * K * 2.0 ** -24 * mag + 1e-30).all())
        assert torch.equal(y.t[:, :N], first.to(dtype))


def test_one_workspace_for_all_arrangements_one_after_the_other():
    cases = []
    for shapes in SHAPES.values():
        for (M, N, K, symmetric) in shapes[:2]:
            *_, x8, s_x, tw = _layer(M, N, K, symmetric)
            own = binding.linear_tiled(x8, s_x, tw, out_dtype=binding.OUT_FP32, workspace=binding.new_workspace(M, N, K, tw.fmt))
            cases.append((x8, s_x, tw, own, torch.empty_like(own)))
    shared = torch.zeros((binding.linear_workspace_bytes(129, 1024, 1024, weight_format=binding.FMT_TILED),), dtype=torch.uint8, device="cuda")
    for _ in range(3):
        for x8, s_x, tw, own, y in cases + cases[::-1]:
            binding.linear_tiled(x8, s_x, tw, out_dtype=binding.OUT_FP32, out=y.zero_(), workspace=shared)
        for *_, own, y in cases:
            assert torch.equal(y, own)
    assert binding.query_device_status() == 0
    assert not bool(shared[:CTL].any())
