"""Host-side checks of csrc/w4a8_decode_plan.h, compiled here with the host compiler: what linear_rows_kernel's waits and memory
rely on holds for every plan, every row and k-block is taken once, without a number of SMs there is no plan, and the shapes of the
GPU tests take the kernels they stand for."""
import ctypes
import os
import random
import subprocess

import pytest

from paper_2505_14638_b200 import build
from decode_shapes import KINDS, RESIDENT, SHAPES, SMS
from test_gpu_rows import ROWS as ROWS_FULL, ROWS_HALF, ROWS_SIGNMAG

NONE, DIRECT, WHOLE, CLUSTER, ROWS, HALF = range(6)
TILED, SIGNMAG = 1, 2

SHIM = r"""
#include "w4a8_decode_plan.h"
using namespace w4a8;
extern "C" int route(long long M, long long N, long long K, int fmt, int sms, int workspace, int on_host, const int* resident, DecodePlan* plan) {
    return decode_choice(M, N, K, fmt, sms, workspace != 0, on_host != 0, [&](int size) { return resident[size]; }, plan);
}
template <class S>
static void put(int* out) {
    const int v[] = {S::G, S::kTmemCols, S::kSmemBudget, S::kFixed, S::kMeta};
    for (int i = 0; i < 5; ++i) out[i] = v[i];
}
extern "C" void sizes(int fmt, int half, int* out) {
    if (fmt == kFmtTiled) half ? put<RowsSizes<kFmtTiled, true>>(out) : put<RowsSizes<kFmtTiled>>(out);
    else half ? put<RowsSizes<kFmtTiledSignMag, true>>(out) : put<RowsSizes<kFmtTiledSignMag>>(out);
}
"""


class DirPlan(ctypes.Structure):
    _fields_ = [(n, ctypes.c_int) for n in ("P", "Wq", "Tc", "xpitch")]


class RowsPlan(ctypes.Structure):
    _fields_ = [(n, ctypes.c_int) for n in ("T", "cut", "units", "more", "RB", "MN", "S1", "S2", "whalf", "smem")]


class DecodePlan(ctypes.Structure):
    _fields_ = [("direct", DirPlan), ("rows", RowsPlan), ("cluster", ctypes.c_int)]


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("decode_plan")
    src, so = d / "plan.cpp", d / "plan.so"
    src.write_text(SHIM)
    subprocess.run([os.environ.get("CXX", "g++"), "-std=c++17", "-O2", "-fPIC", "-shared", "-I" + build.CSRC, "-o", str(so), str(src)],
                   check=True, capture_output=True)
    lib = ctypes.CDLL(str(so))
    lib.route.argtypes = [ctypes.c_longlong] * 3 + [ctypes.c_int] * 4 + [ctypes.c_void_p, ctypes.c_void_p]
    return lib


def _route(lib, M, N, K, fmt, sms=SMS, workspace=True, on_host=False, resident=RESIDENT):
    plan = DecodePlan()
    return lib.route(M, N, K, fmt, sms, workspace, on_host, (ctypes.c_int * 9)(*resident), ctypes.byref(plan)), plan


def _shapes():
    rng = random.Random(7)
    for _ in range(4000):
        N, K = 16 * int(2 ** rng.uniform(0, 12)), 128 * int(2 ** rng.uniform(0, 7.2))
        yield rng.randint(1, 16) if rng.random() < 0.6 else rng.randint(17, 128), N, K, rng.choice((TILED, SIGNMAG)), rng.random() < 0.8


def test_plans_of_rows_hold_what_the_kernel_relies_on(lib):
    seen = set()
    for M, N, K, fmt, workspace in _shapes():
        for resident in (RESIDENT, [-1] * 9):
            kind, plan = _route(lib, M, N, K, fmt, workspace=workspace, resident=resident)
            assert kind != NONE
            if kind not in (ROWS, HALF):
                continue
            p = plan.rows
            v = (ctypes.c_int * 5)()
            lib.sizes(fmt, int(kind == HALF), v)
            G, cols, budget, fixed, meta = v
            what = (M, N, K, fmt, workspace, kind)
            ks, runs = 2 // p.RB, p.T // p.cut
            assert p.T == runs * p.cut and runs * p.units + p.more == N // 8 and 0 <= p.more < runs, what
            rows = 8 * (p.units + (p.more > 0))
            assert rows <= 128 * p.RB and p.RB in (1, 2) and p.MN % 16 == 0 and M <= p.MN < M + 16, what
            # a slot of expanded weights per expansion group, and weights landed ahead of every slot
            assert G <= p.S2 <= 8 and p.S2 <= p.S1 <= 16, what
            assert (p.RB * p.MN + 31) // 32 * 32 + 64 * p.S2 <= cols, what
            assert p.whalf >= rows * (64 + meta) and p.whalf % 128 == 0, what
            assert p.smem == fixed + p.S2 * ks * p.MN * 128 + p.S1 * ks * p.whalf <= budget, what
            if p.cut > 1:   # a CTA per part; counters per run and partial sums in the workspace
                assert M <= 16 and workspace and p.T <= SMS and p.RB == 1 and K // 128 >= 4 * p.cut, what
            seen.add((kind, p.cut > 1, p.RB, p.T > SMS))
    assert {(ROWS, True, 1, False), (ROWS, False, 2, False), (ROWS, False, 2, True), (HALF, False, 1, False),
            (HALF, True, 1, False)} <= seen


@pytest.mark.parametrize("M,N,K", [(1, 4096, 4096), (8, 1024, 1024), (16, 28672, 4096), (32, 4096, 4096), (128, 28672, 4096)])
def test_no_number_of_sms_is_an_error_and_not_a_division(lib, M, N, K):
    for sms in (0, -1):
        for workspace in (True, False):
            assert _route(lib, M, N, K, SIGNMAG, sms=sms, workspace=workspace)[0] == NONE


@pytest.mark.parametrize("kind", sorted(SHAPES))
def test_shapes_of_the_gpu_tests_take_the_kernels_they_stand_for(lib, kind):
    rings = set()
    for M, N, K, symmetric in SHAPES[kind]:
        got, plan = _route(lib, M, N, K, SIGNMAG if symmetric else TILED, resident=RESIDENT)
        assert KINDS[got] == kind, (M, N, K, symmetric, KINDS[got])
        rings.add((plan.rows.RB, plan.rows.S1, plan.rows.S2, plan.rows.cut > 1, plan.rows.T > SMS))
    if kind == "rows":
        assert (1, 4, 4, False, False) in rings and {r[3:] for r in rings} == {(True, False), (False, False), (False, True)}
    if kind == "rows_half":
        assert {r[3:] for r in rings} == {(True, False), (False, False), (False, True)}


@pytest.mark.parametrize("fmt", [SIGNMAG, TILED])
def test_the_shapes_of_rows_take_rows(lib, fmt):
    for want, shapes in ((ROWS, ROWS_FULL), (HALF, ROWS_HALF), (ROWS if fmt == SIGNMAG else WHOLE, ROWS_SIGNMAG)):
        assert [(s, _route(lib, *s, fmt)[0]) for s in shapes] == [(s, want) for s in shapes]


def test_without_a_workspace_k_is_not_cut(lib):
    for M, N, K, fmt, _ in _shapes():
        kind, plan = _route(lib, M, N, K, fmt, workspace=False)
        assert M > 16 or kind == WHOLE or plan.rows.cut == 1
