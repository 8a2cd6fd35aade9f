"""GPU: the quantizer's persistent kernel where its order of tasks, its tile loads and its marks can go wrong: panels of eight blocks,
rows behind the last complete group of four with U at a base that tile loads cannot read, calls on two streams at once, a call
replayed from a graph (marks in buffers that hold the results of the call before)."""
import pytest
import torch

from paper_2505_14638_b200 import binding

pytestmark = pytest.mark.gpu


def _layer(N, K, offset=0, seed=0):
    g = torch.Generator(device="cuda")
    g.manual_seed(N + K + seed)
    W = torch.randn((N, K), generator=g, device="cuda") * 0.02
    buf = torch.empty((K * K + 4,), device="cuda")
    U = buf[offset:offset + K * K].view(K, K)
    U.copy_(torch.eye(K, device="cuda") + 0.5 * torch.triu(torch.randn((K, K), generator=g, device="cuda"), 1) / K ** 0.5)
    return W, U, binding.gar_permutation(torch.rand(K, generator=g, device="cuda"))


def _same(a, b, rows=slice(None)):
    return all(torch.equal(x[rows].contiguous().view(torch.uint8), y.contiguous().view(torch.uint8)) for x, y in zip(a, b) if x is not None)


@pytest.mark.parametrize("N,K,offset", [(8192, 4224, 0), (8195, 4096, 1), (1157, 1408, 3), (1, 1024, 0), (2, 384, 1)])
def test_rows_in_slabs(N, K, offset):
    # rows do not depend on one another (per-channel scales): slabs of 64 rows take one block's errors at a time throughout
    W, U, perm = _layer(N, K, offset)
    whole = binding.dpq_quantize(W, U, perm, symmetric=False, mse_steps=2, per_channel=True)
    for r0 in sorted({0, min(128, N - 1), max(N - 64, 0), max(N - 3, 0)}):
        rows = slice(r0, min(r0 + 64, N))
        slab = binding.dpq_quantize(W[rows].contiguous(), U.clone(), perm, symmetric=False, mse_steps=2, per_channel=True)
        assert _same(whole, slab, rows)
    assert binding.query_device_status() == 0


def test_two_streams_and_a_graph():
    layers = [_layer(1024, 2048, seed=i) for i in range(2)]
    want = [binding.dpq_quantize(*l, symmetric=True, mse_steps=6) for l in layers]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(2)]
    for rep in range(5):
        got = []
        for l, s in zip(layers, streams):
            with torch.cuda.stream(s):
                got.append(binding.dpq_quantize(*l, symmetric=True, mse_steps=6))
        torch.cuda.synchronize()
        assert all(_same(a, b) for a, b in zip(want, got)), rep
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        out = binding.dpq_quantize(*layers[0], symmetric=True, mse_steps=6)
    for rep in range(4):
        g.replay()
        torch.cuda.synchronize()
        assert _same(want[0], out), rep
    assert binding.query_device_status() == 0
