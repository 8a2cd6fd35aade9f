"""GPU: launches that start while an earlier kernel of the stream is still running (programmatic stream
serialization) must not count its run time against the limit of their bounded waits.  The earlier kernel
releases its dependents at once and returns after 2.3 s, more than the limit of two seconds; the
launch behind it must then return the same bits as an undisturbed one and leave the status word clean.  One
shape per kernel and plan, each with more k-blocks per CTA than its rings hold, so that every role gets
to wait."""
import ctypes
import subprocess

import pytest
import torch

from paper_2505_14638_b200 import binding, build

pytestmark = pytest.mark.gpu

HOLD = r"""
__global__ void hold(unsigned long long ns) {
    asm volatile("griddepcontrol.launch_dependents;");
    unsigned long long t0, t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
    for (int i = 0; i < 20000; ++i) {   // (at most 20000 naps of up to a millisecond)
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
        if (t - t0 >= ns) break;
        __nanosleep(500000);
    }
}
extern "C" int run_hold(unsigned long long ns, void* stream) {
    hold<<<1, 32, 0, static_cast<cudaStream_t>(stream)>>>(ns);
    return static_cast<int>(cudaGetLastError());
}
"""


@pytest.fixture(scope="module")
def hold(tmp_path_factory):
    d = tmp_path_factory.mktemp("hold")
    src, so = d / "hold.cu", d / "hold.so"
    src.write_text(HOLD)
    cmd = [a for a in build.nvcc_command(str(so)) if a not in build.SOURCES] + [str(src)]
    subprocess.run(cmd, check=True, capture_output=True)
    f = ctypes.CDLL(str(so)).run_hold
    f.argtypes = [ctypes.c_ulonglong, ctypes.c_void_p]
    return f


def _layer(M, N, K, fmt, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    W = torch.randn((N, K), generator=g, device="cuda") * 0.02
    wq = binding.quantize_weight_rtn(W, symmetric=fmt != binding.FMT_TILED)
    x = torch.randn((M, K), generator=g, device="cuda").to(torch.bfloat16)
    return x, wq, wq if fmt == binding.FMT_CANONICAL else binding.prepack_weight(*wq)


def _linear(M, N, K, fmt):
    x, _, w = _layer(M, N, K, fmt, M + N + K)
    x8, s_x = binding.quantize_act(x)
    ws = binding.new_workspace(M, N, K, fmt)
    y = torch.empty((M, N), device="cuda")
    if fmt == binding.FMT_CANONICAL:
        return y, lambda: binding.linear(x8, s_x, *w, out_dtype=binding.OUT_FP32, out=y, workspace=ws)
    return y, lambda: binding.linear_tiled(x8, s_x, w, out_dtype=binding.OUT_FP32, out=y, workspace=ws)


def _chain():
    layers = [_layer(8, 8192, 4096, binding.FMT_TILED_SIGNMAG, 5), _layer(16, 14336, 2048, binding.FMT_TILED_SIGNMAG, 6)]
    y = torch.empty((24, 14336), device="cuda")
    probs = [dict(x=layers[0][0], weight=layers[0][2], y=y[:8, :8192]), dict(x=layers[1][0], weight=layers[1][2], y=y[8:])]
    return y, binding.LinearChain(probs)


def _w4a16():
    x, _, w = _layer(600, 4096, 4096, binding.FMT_TILED_SIGNMAG, 7)
    y = torch.empty((600, 4096), device="cuda")
    return y, lambda: binding.linear_w4a16_tiled(x, w, out=y, out_dtype=binding.OUT_FP32)


def _w8a8():
    x, wq, _ = _layer(2400, 2048, 2048, binding.FMT_CANONICAL, 8)
    w8 = binding.dequant_weight(*wq[:3])
    x8, s_x = binding.quantize_act(x)
    y = torch.empty((2400, 2048), device="cuda")
    return y, lambda: binding.linear_w8a8(x8, s_x, w8, wq[3], out_dtype=binding.OUT_FP32, out=y)


SM, TI, CA = binding.FMT_TILED_SIGNMAG, binding.FMT_TILED, binding.FMT_CANONICAL
CASES = {
    "runs of rows": lambda: _linear(8, 14336, 4096, SM),
    "runs of rows, K cut": lambda: _linear(8, 4096, 14336, TI),
    "runs of rows, half an SM": lambda: _linear(8, 14336, 1536, SM),
    "runs of rows, half an SM, K cut": lambda: _linear(8, 4096, 4096, TI),
    "whole tiles, 128 tokens, wide layer": lambda: _linear(100, 28672, 2048, TI),
    "runs of rows, 128 tokens": lambda: _linear(100, 28672, 8192, SM),
    "cluster, 64 tokens": lambda: _linear(40, 4096, 14336, SM),
    "K cut between CTAs, 128 tokens, generic": lambda: _linear(130, 1024, 14336, TI),
    "K cut between CTAs, 128 tokens": lambda: _linear(300, 1024, 14336, SM),
    "K cut between CTAs, 256 tokens": lambda: _linear(193, 4000, 14336, TI),
    "whole tiles, 64 tokens": lambda: _linear(200, 4080, 4096, SM),
    "whole tiles, 256 tokens": lambda: _linear(1196, 3680, 4864, TI),
    "pairs, K cut": lambda: _linear(512, 4096, 14336, TI),
    "pairs, 256 x 256 tiles": lambda: _linear(2048, 4096, 4096, SM),
    "pairs, 256 x 256 tiles, wide layer": lambda: _linear(1100, 16384, 2048, SM),
    "pairs, 256 x 512 tiles": lambda: _linear(1152, 7648, 2560, TI),
    "canonical": lambda: _linear(100, 14336, 4096, CA),
    "chain": _chain,
    "W4A16": _w4a16,
    "W8A8": _w8a8,
}


@pytest.mark.parametrize("case", CASES)
def test_time_of_an_earlier_kernel_does_not_count(hold, case):
    y, run = CASES[case]()
    y.fill_(float("nan"))
    run()
    torch.cuda.synchronize()
    assert binding.query_device_status() == 0
    want = y.clone()
    assert not bool(want[:8, :8192].isnan().any())
    y.fill_(float("nan"))
    torch.cuda.synchronize()
    assert hold(2_300_000_000, torch.cuda.current_stream().cuda_stream) == 0
    run()
    torch.cuda.synchronize()
    assert binding.query_device_status() == 0
    assert torch.equal(y.view(torch.int32), want.view(torch.int32))
