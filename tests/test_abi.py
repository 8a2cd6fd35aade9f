"""Host-side checks of the C-ABI library: it loads, exports what include/w4a8.h declares, and
rejects bad arguments before touching a device (no GPU needed)."""
import ctypes
import os
import re
import sys

import pytest

from paper_2505_14638_b200 import binding, build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def L():
    build.build()
    return binding.lib()


def test_exports_every_declared_symbol(L):
    hdr = open(os.path.join(ROOT, "include", "w4a8.h")).read()
    hdr = re.sub(r"/\*.*?\*/", "", hdr, flags=re.S)
    declared = set(re.findall(r"\b(w4a8_[a-z0-9_]+)\s*\(", hdr))
    assert declared == set(binding.EXPORTS)
    for name in declared:
        assert hasattr(L, name), name
    assert 'extern "C"' in open(os.path.join(ROOT, "include", "w4a8.h")).read()


def test_status_strings(L):
    assert binding.status_string(0) == "ok"
    for code in range(-7, 0):
        assert binding.status_string(code) not in ("ok", "unknown status")
    assert binding.status_string(-99) == "unknown status"


def test_workspace_and_prepack_size_queries_are_host_only(L):
    assert L.w4a8_prepack_bytes(14336, 4096, binding.FMT_TILED_SIGNMAG) == 14336 * 32 * 66
    assert L.w4a8_prepack_bytes(14336 + 16, 4096, binding.FMT_TILED) == (14336 + 16) * 32 * 68
    assert L.w4a8_prepack_bytes(14336, 4096, binding.FMT_CANONICAL) == 0
    assert binding.linear_workspace_bytes(16, 14336, 4096, weight_format=binding.FMT_TILED_SIGNMAG) == 65536 + 160 * 128 * 128 * 4   # control area of fixed size (counters), partial tiles
    ws = binding.linear_workspace_bytes(2048, 4096, 4096, weight_format=binding.FMT_TILED_SIGNMAG)
    assert ws >= 2 * 8 * 32 * 4 + 2 * 148 * 256 * 128 * 4
    assert binding.linear_workspace_bytes(2048, 4096, 4096) == 0          # large M: no split
    ws = binding.linear_workspace_bytes(16, 14336, 4096)
    assert ws % (16 * 14336 * 4) == 0 and ws > 0                          # S partial tiles
    assert binding.linear_workspace_bytes(16, 14336, 4096, binding.ALGO_UMMA, 4) == 4 * 16 * 14336 * 4
    assert binding.linear_workspace_bytes(16, 14336, 4096, binding.ALGO_SIMT, 0) == 0
    assert binding.linear_workspace_bytes(16, 14336, 100) == 0            # invalid K


def _fake(addr=0x1000):
    return ctypes.c_void_p(addr)


def test_quantize_act_rejects_bad_arguments(L):
    p = _fake()
    f = L.w4a8_quantize_act
    assert f(None, 4, 128, 128, p, 128, p, 0, None, None) == binding.ERR_INVALID_ARG
    assert f(p, 0, 128, 128, p, 128, p, 0, None, None) == binding.ERR_INVALID_ARG
    assert f(p, 4, 128, 128, p, 128, p, 7, None, None) == binding.ERR_INVALID_ARG
    assert f(p, 4, 100, 128, p, 128, p, 0, None, None) == binding.ERR_BAD_SHAPE
    assert f(p, 4, 128, 64, p, 128, p, 0, None, None) == binding.ERR_BAD_SHAPE
    assert f(_fake(0x1004), 4, 128, 128, p, 128, p, 0, None, None) == binding.ERR_BAD_ALIGNMENT
    assert f(p, 4, 128, 132, p, 128, p, 0, None, None) == binding.ERR_BAD_ALIGNMENT


def test_dequant_rejects_bad_arguments(L):
    p = _fake()
    f = L.w4a8_dequant_weight
    assert f(None, p, None, 16, 128, 128, p, None) == binding.ERR_INVALID_ARG
    assert f(p, p, None, 16, 128, 64, p, None) == binding.ERR_BAD_SHAPE
    assert f(p, p, None, 16, 192, 128, p, None) == binding.ERR_BAD_SHAPE
    assert f(_fake(0x1008), p, None, 16, 128, 128, p, None) == binding.ERR_BAD_ALIGNMENT


def test_linear_rejects_bad_arguments(L):
    p = _fake()
    f = L.w4a8_linear

    def call(x8=p, ldx8=4096, s_x=p, M=16, codes=p, gs=p, gz=None, fmt=0, s_w=p, sws=0, N=14336, K=4096,
             group=128, y=p, ldy=14336, od=0, ws=p, wsb=1 << 30):
        return f(x8, ldx8, s_x, M, codes, gs, gz, fmt, s_w, sws, N, K, group, y, ldy, od, ws, wsb, None)

    assert call(fmt=3) == binding.ERR_INVALID_ARG
    assert call(gs=None) == binding.ERR_INVALID_ARG
    assert call(fmt=2, gs=None, M=512, ws=None, wsb=0) == binding.ERR_WORKSPACE_TOO_SMALL
    assert call(fmt=1, gs=None, M=512, wsb=1024) == binding.ERR_WORKSPACE_TOO_SMALL

    assert call(x8=None) == binding.ERR_INVALID_ARG
    assert call(M=0) == binding.ERR_INVALID_ARG
    assert call(sws=2) == binding.ERR_INVALID_ARG
    assert call(od=5) == binding.ERR_INVALID_ARG
    assert call(K=4000) == binding.ERR_BAD_SHAPE
    assert call(group=64) == binding.ERR_BAD_SHAPE
    assert call(N=14337, ldy=14352) == binding.ERR_BAD_SHAPE
    assert call(ldx8=2048) == binding.ERR_BAD_SHAPE
    assert call(ldy=1024) == binding.ERR_BAD_SHAPE
    assert call(x8=_fake(0x1001)) == binding.ERR_BAD_ALIGNMENT
    assert call(ldx8=4100) == binding.ERR_BAD_ALIGNMENT
    assert call(ws=None, wsb=0) == binding.ERR_WORKSPACE_TOO_SMALL
    assert call(wsb=16) == binding.ERR_WORKSPACE_TOO_SMALL
    g = L.w4a8_linear_ex
    assert g(p, 4096, p, 16, p, p, None, p, 0, 14336, 4096, 128, p, 14336, 0, p, 1 << 30, 9, 0, None) \
        == binding.ERR_INVALID_ARG
    assert g(p, 4096, p, 16, p, p, None, p, 0, 14336, 4096, 128, p, 14336, 0, p, 1 << 30, 2, 5, None) \
        == binding.ERR_BAD_SHAPE                                            # 5 does not divide K/128


def test_rtn_and_host_forward_reject_bad_arguments(L):
    p = _fake()
    f = L.w4a8_quantize_weight_rtn
    assert f(None, 16, 128, 128, 1, 0, 0, p, p, None, p, None) == binding.ERR_INVALID_ARG
    assert f(p, 16, 128, 128, 0, 0, 0, p, p, None, p, None) == binding.ERR_INVALID_ARG   # asymmetric needs gzero
    assert f(p, 16, 130, 128, 1, 0, 0, p, p, None, p, None) == binding.ERR_BAD_SHAPE
    h = L.w4a8_forward_host
    assert h(None, 4, p, p, None, 0, p, 0, 16, 128, 128, p, p, p, p, p, None, 0, None) == binding.ERR_INVALID_ARG
    assert h(p, 4, p, p, None, 0, p, 0, 16, 100, 128, p, p, p, p, p, None, 0, None) == binding.ERR_BAD_SHAPE
    assert h(p, 4, p, p, None, 9, p, 0, 16, 128, 128, p, p, p, p, p, None, 0, None) == binding.ERR_INVALID_ARG
    k = L.w4a8_prepack_weight
    assert k(None, p, None, 16, 128, 128, 1, p, 1 << 20, None) == binding.ERR_INVALID_ARG
    assert k(p, p, None, 16, 128, 128, 0, p, 1 << 20, None) == binding.ERR_INVALID_ARG      # canonical is not a target
    assert k(p, p, p, 16, 128, 128, 2, p, 1 << 20, None) == binding.ERR_INVALID_ARG          # sign-magnitude needs z = 8
    assert k(p, p, None, 16, 100, 128, 1, p, 1 << 20, None) == binding.ERR_BAD_SHAPE
    assert k(p, p, None, 16, 128, 128, 1, _fake(0x1010), 1 << 20, None) == binding.ERR_BAD_ALIGNMENT
    assert k(p, p, None, 16, 128, 128, 1, p, 100, None) == binding.ERR_WORKSPACE_TOO_SMALL
    assert L.w4a8_query_device_status(None) == binding.ERR_INVALID_ARG


def test_missing_library_fails_loudly(monkeypatch, tmp_path):
    monkeypatch.setattr(binding, "_lib", None)
    monkeypatch.setattr(binding, "LIB_PATH", str(tmp_path / "nope.so"))
    with pytest.raises(RuntimeError, match="no fallback"):
        binding.lib()


def test_extension_module_marshals_and_refuses(L):
    # sizes agree with the ctypes route; arguments that are not tensors, or not as many, raise; CPU tensors are refused
    # before anything is launched; a status of the library comes back as one
    import torch
    h = binding._load_host()
    for M, N, K, fmt in ((16, 14336, 4096, 0), (2048, 4096, 4096, 0), (5, 1024, 1024, 2), (16, 14336, 100, 0)):
        assert h.linear_workspace_bytes(M, N, K, fmt) == int(L.w4a8_linear_workspace_bytes(M, N, K, fmt))
    x = torch.zeros((4, 128), dtype=torch.bfloat16)
    with pytest.raises(AssertionError):
        h.quantize_act(x, x, x, 0, None)
    with pytest.raises(TypeError):
        h.quantize_act(x, 1, x, 0, None)
    with pytest.raises(TypeError):
        h.quantize_act(x)
    x8 = torch.zeros((4, 128), dtype=torch.uint8)
    s = torch.ones(1)
    with pytest.raises(AssertionError):   # K differs
        h.linear(x8, s, x8, None, None, binding.FMT_TILED, s, 16, 256, 128, s, 0, None)


class _Wrapped:
    """A buffer that is not a torch tensor: what it knows it asks the tensor it holds."""

    def __init__(self, t):
        self._t = t

    def __getattr__(self, name):
        return getattr(self._t, name)


def test_buffers_that_are_not_torch_tensors_reach_the_library(L, monkeypatch):
    # (addresses that are not 16-byte aligned: the library refuses them before it touches a device)
    import torch
    monkeypatch.setattr(binding, "_stream", lambda: None)
    raw = torch.zeros(4 * 128 + 32, dtype=torch.uint8)
    at = 1 + (-raw.data_ptr()) % 16
    x8, s, out = raw[at:at + 4 * 128].view(4, 128), torch.ones(4), torch.zeros((4, 16), dtype=torch.bfloat16)
    w = torch.zeros(16 * 128, dtype=torch.uint8)
    tw = binding.TiledWeight(_Wrapped(w), binding.FMT_TILED, 16, 128, _Wrapped(torch.ones(1)))
    codes, gs = _Wrapped(torch.zeros((16, 64), dtype=torch.uint8)), _Wrapped(torch.ones((16, 1), dtype=torch.bfloat16))
    for call in (lambda: binding.linear_tiled(_Wrapped(x8), _Wrapped(s), tw, out=_Wrapped(out), workspace=_Wrapped(raw)),
                 lambda: binding.linear(_Wrapped(x8), _Wrapped(s), codes, gs, None, _Wrapped(s[:1]), out=_Wrapped(out),
                                        workspace=_Wrapped(torch.zeros(1 << 20, dtype=torch.uint8)))):
        with pytest.raises(binding.W4A8Error) as e:
            call()
        assert binding.status_string(binding.ERR_BAD_ALIGNMENT) in str(e.value)
    with pytest.raises(AssertionError):      # not on the device
        binding.quantize_act(_Wrapped(torch.zeros((4, 128), dtype=torch.bfloat16)), out=(_Wrapped(x8), _Wrapped(s)))
    with pytest.raises(AttributeError):      # not a buffer at all
        binding.linear_tiled(3, s, tw, out=out, workspace=raw)


def test_the_c_library_builds_without_torch(L, monkeypatch, tmp_path):
    # (the library itself is there; the extension module would have to be built)
    monkeypatch.setattr(build, "HOST_PATH", str(tmp_path / "_w4a8_host.so"))
    monkeypatch.setattr(build, "host_command", lambda out: pytest.fail("needs torch"))
    monkeypatch.setitem(sys.modules, "torch", None)      # import torch raises ImportError
    assert build.build() == build.LIB_PATH
    assert not os.path.exists(build.HOST_PATH)


def test_the_extension_module_is_built_again_for_another_torch(L, monkeypatch):
    import torch
    assert torch.__version__ in binding._load_host().__doc__
    built = []
    monkeypatch.setattr(build, "_run", lambda cmd, out, *a: built.append(out))
    build.build()
    assert built == []
    monkeypatch.setattr(torch, "__version__", "99.0")
    build.build()
    assert built == [build.HOST_PATH]


@pytest.mark.parametrize("M,N,K", [(33, 6144, 4096), (64, 1024, 4096), (17, 144, 8192), (8, 1024, 1024), (16, 4096, 2048)])
def test_no_workspace_is_asked_for_where_none_is_used(L, M, N, K):
    # canonical weights, kernel chosen by the library; the kernel that cuts K through the workspace still asks for it
    assert L.w4a8_linear_workspace_bytes(M, N, K, binding.FMT_CANONICAL) == 0
    assert L.w4a8_linear_ex_workspace_bytes(M, N, K, binding.ALGO_AUTO, 0) == 0
    assert L.w4a8_linear_ex_workspace_bytes(M, N, K, binding.ALGO_UMMA, 0) > 0
    assert L.w4a8_linear_workspace_bytes(16, 14336, 4096, binding.FMT_CANONICAL) > 0
