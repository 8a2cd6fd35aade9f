"""Builds the CUDA library in-tree with nvcc for sm_100a, and, where torch is installed, the binding's per-layer
calls (a small extension module against torch's headers) with the host compiler.  No JIT cache.
`--library-only` builds the C-ABI library alone, which needs nvcc and nothing else."""
from __future__ import annotations

import os
import subprocess
import sys

_HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(_HERE, "csrc")
LIB_PATH = os.path.join(_HERE, "libw4a8_b200.so")
HOST_PATH = os.path.join(_HERE, "_w4a8_host.so")
SOURCES = [os.path.join(CSRC, "w4a8_lib.cu")]
HOST_SOURCE = os.path.join(CSRC, "w4a8_host.cpp")


def _deps():
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if not f.endswith(".cpp")]
    deps.append(os.path.join(os.path.dirname(_HERE), "include", "w4a8.h"))
    return deps


def nvcc_command(out_path: str, verbose: bool = False):
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    cmd = [
        nvcc, "-std=c++17", "-O3", "-lineinfo",
        "-gencode", "arch=compute_100a,code=sm_100a",
        "-Xcompiler", "-fPIC", "-shared",
        "-o", out_path,
    ]
    if verbose:
        cmd += ["-Xptxas", "-v"]
    return cmd + SOURCES + ["-lcudart"]


def host_versions() -> str:
    """What the extension module is compiled against; it carries this text."""
    import torch
    return "torch %s, Python %d.%d" % (torch.__version__, sys.version_info[0], sys.version_info[1])


def host_command(out_path: str):
    import sysconfig

    import torch
    root = os.path.dirname(torch.__file__)
    cuda = os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")))
    return [
        os.environ.get("CXX", "g++"), "-std=c++17", "-O2", "-fPIC", "-shared", "-fvisibility=hidden",
        "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI),
        '-DW4A8_HOST_VERSIONS="%s"' % host_versions(),
        "-I" + os.path.join(root, "include"), "-I" + os.path.join(root, "include", "torch", "csrc", "api", "include"),
        "-I" + os.path.join(cuda, "include"), "-I" + sysconfig.get_paths()["include"],
        "-o", out_path, HOST_SOURCE,
        "-L" + os.path.join(root, "lib"), "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda",
        "-L" + _HERE, "-l:" + os.path.basename(LIB_PATH), "-Wl,-rpath,$ORIGIN",
    ]


def _run(cmd, out, tmp, what, verbose=False):
    res = subprocess.run(cmd, capture_output=True, text=True)
    if verbose:
        sys.stderr.write(res.stderr)
    if res.returncode != 0:
        raise RuntimeError(what + " failed:\n" + res.stdout + res.stderr)
    os.replace(tmp, out)


def _stale(out, deps):
    return not os.path.exists(out) or any(os.path.getmtime(d) > os.path.getmtime(out) for d in deps)


def _built_against(path, versions):
    with open(path, "rb") as f:
        return (versions + "\0").encode() in f.read()


def _has_torch():
    try:
        import torch  # noqa: F401
    except ImportError:
        return False
    return True


def build_library(force: bool = False, verbose: bool = False) -> str:
    """The C-ABI library alone."""
    if force or _stale(LIB_PATH, _deps()):
        tmp = LIB_PATH + ".tmp%d" % os.getpid()
        _run(nvcc_command(tmp, verbose), LIB_PATH, tmp, "nvcc", verbose)
    return LIB_PATH


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile what is missing or older than a source. Returns the CUDA library's path."""
    build_library(force, verbose)
    if not _has_torch():
        sys.stderr.write("torch is not installed: the C library is complete, the Python binding's extension module is not built\n")
        return LIB_PATH
    if force or _stale(HOST_PATH, [HOST_SOURCE, _deps()[-1]]) or not _built_against(HOST_PATH, host_versions()):
        tmp = HOST_PATH + ".tmp%d" % os.getpid()
        _run(host_command(tmp), HOST_PATH, tmp, "g++")
    return LIB_PATH


if __name__ == "__main__":
    make = build_library if "--library-only" in sys.argv else build
    print(make(force="--force" in sys.argv, verbose="-v" in sys.argv))
