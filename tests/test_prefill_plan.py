"""Host-side checks of csrc/w4a8_prefill_plan.h, compiled here with the host compiler: the tile order of CTA pairs visits
every tile once, and the rounds that the cost model counts are those of the schedule (a model that counted half a round
for tiles which the order mixed with whole ones chose 256 x 512 tiles where they took up to 1.3 times the time of the
next alternative, (1152, 7648, 2560) for one); the shapes of the GPU tests take the arrangements they stand for."""
import ctypes
import os
import random
import subprocess

import pytest

from paper_2505_14638_b200 import build
from prefill_shapes import KINDS, QUADS, SHAPES, SMS

SHIM = r"""
#include "w4a8_prefill_plan.h"
using namespace w4a8;
extern "C" long long half_rounds(long long M, long long N, long long pairs) {
    return 2 * pair_rounds(M, N, pairs, true) + pair_rounds(M, N, pairs, false);
}
extern "C" void tiles(long long M, long long N, int tokens, int* nt, int* mt) {
    const int TM = (int)((M + tokens - 1) / tokens), TN = (int)((N + 255) / 256);
    for (int t = 0; t < TM * TN; ++t) pair_tile(t, pair_full_tiles(M, tokens, TM), TN, nt[t], mt[t]);
}
extern "C" int choice(long long M, long long N, long long K, int signmag, int sms, int quads, SkPlan* pl) {
    return prefill_choice(M, N, K, signmag != 0, sms, quads, pl);
}
"""


class SkPlan(ctypes.Structure):
    _fields_ = [("bnx", ctypes.c_int), ("TM", ctypes.c_int), ("TN", ctypes.c_int), ("per", ctypes.c_int), ("P", ctypes.c_int64),
                ("counter_bytes", ctypes.c_size_t)]


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    src, so = d / "plan.cpp", d / "plan.so"
    src.write_text(SHIM)
    subprocess.run([os.environ.get("CXX", "g++"), "-std=c++17", "-O2", "-fPIC", "-shared", "-I" + build.CSRC, "-o", str(so), str(src)],
                   check=True, capture_output=True)
    lib = ctypes.CDLL(str(so))
    lib.half_rounds.argtypes, lib.half_rounds.restype = [ctypes.c_longlong] * 3, ctypes.c_longlong
    lib.choice.argtypes = [ctypes.c_longlong] * 3 + [ctypes.c_int] * 3 + [ctypes.POINTER(SkPlan)]
    lib.tiles.argtypes = [ctypes.c_longlong, ctypes.c_longlong, ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p]
    return lib


def _tiles(plan, M, N, tokens):
    n = -(-M // tokens) * -(-N // 256)
    nt, mt = (ctypes.c_int * n)(), (ctypes.c_int * n)()
    plan.tiles(M, N, tokens, nt, mt)
    return list(zip(nt, mt))


def _shapes():
    rng = random.Random(5)
    named = [(1152, 7648), (526, 14128), (700, 12304), (8192, 28672), (4609, 9488), (513, 18448), (256, 28672), (257, 256)]
    return named + [(rng.randint(129, 9000), 16 * rng.randint(1, 1800)) for _ in range(200)]


@pytest.mark.parametrize("tokens", [256, 512])
def test_every_tile_once(plan, tokens):
    for M, N in _shapes():
        got = _tiles(plan, M, N, tokens)
        assert sorted(got) == sorted((n, m) for n in range(-(-N // 256)) for m in range(-(-M // tokens))), (M, N)


@pytest.mark.parametrize("pairs", [74, 66, 1])
def test_rounds_of_the_model_are_those_of_the_schedule(plan, pairs):
    for M, N in _shapes():
        cost = [2 if M - 512 * m > 256 else 1 for _, m in _tiles(plan, M, N, 512)]
        assert plan.half_rounds(M, N, pairs) == max(sum(cost[c::pairs]) for c in range(min(pairs, len(cost)))), (M, N)


def _choice(plan, M, N, K, signmag, sms=SMS, quads=QUADS):
    pl = SkPlan()
    return KINDS[plan.choice(M, N, K, int(signmag), sms, quads, ctypes.byref(pl))], pl


@pytest.mark.parametrize("quads", [37, 33, 12, -1])
def test_k_is_cut_between_pairs_in_one_round_only(plan, quads):
    # a cluster of four CTAs works on one tile: no more tiles than clusters that the device holds at once
    rng = random.Random(quads)
    named = [(374, 4608, 11904), (1488, 1376, 10496), (1557, 1280, 7296), (512, 4096, 14336), (300, 2064, 8320), (257, 256, 14336)]
    shapes = named + [(rng.randint(129, 2000), 16 * rng.randint(16, 600), 128 * rng.randint(8, 112)) for _ in range(2000)]
    cut = [(M, N) for M, N, K in shapes if _choice(plan, M, N, K, True, quads=quads)[0] == "pairs_k_cut"]
    assert all(-(-M // 256) * -(-N // 256) <= quads for M, N in cut)
    assert bool(cut) == (quads > 0)


@pytest.mark.parametrize("kind", KINDS)
def test_the_gpu_tests_take_the_arrangements_they_stand_for(plan, kind):
    for M, N, K, symmetric in SHAPES[kind]:
        assert _choice(plan, M, N, K, symmetric)[0] == kind, (M, N, K, symmetric)


@pytest.mark.parametrize("sms", [148, 132, 60])
def test_plans_of_the_persistent_kernel(plan, sms):
    rng = random.Random(sms)
    for _ in range(4000):
        M, N, K = rng.randint(129, 4000), 16 * rng.randint(1, 1800), 128 * rng.randint(1, 112)
        kind, pl = _choice(plan, M, N, K, rng.random() < 0.5, sms)
        if kind.startswith("pairs"):
            continue
        bnx, tiles = int(kind.lstrip("wholecut")), pl.TM * pl.TN
        assert (pl.bnx, pl.TM, pl.TN) == (bnx, -(-M // bnx), -(-N // 128))
        if kind.startswith("whole"):
            assert pl.per == 1 and pl.P == min(tiles, sms)
        else:
            # resident at once, each with k-blocks of its own
            assert pl.P == pl.per * tiles <= sms and 2 <= pl.per <= K // 128 // 2
