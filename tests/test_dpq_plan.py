"""Host-side check of csrc/w4a8_dpq_plan.h, compiled here with the host compiler: the quantizer's tasks come in an order in which each
follows those it waits for (a block's task: the errors of all blocks but the last one before it have been applied to its columns;
an application: the blocks are done, the errors before theirs have been applied), every column sees all errors in ascending
order, and with enough tiles the errors of up to eight blocks go together."""
import ctypes
import os
import subprocess

import pytest

from paper_2505_14638_b200 import build

SHIM = r"""
#include "w4a8_dpq_plan.h"
using namespace w4a8;
extern "C" void steps(int G, int row_tiles, int slots, int* out) {   // per step: far, near as (errors, blocks, first, count)
    DpqSteps s = {};
    s.G = G;
    s.row_tiles = row_tiles;
    s.slots = slots;
    s.b = -1;
    for (int b = 0; b < G; ++b) {
        s.next();
        const DpqTrail t[2] = {s.far, s.near};
        for (int i = 0; i < 2; ++i) {
            const int v[4] = {t[i].errors, t[i].blocks, t[i].first, t[i].count};
            for (int k = 0; k < 4; ++k) *out++ = v[k];
        }
    }
}
"""


@pytest.fixture(scope="module")
def steps(tmp_path_factory):
    d = tmp_path_factory.mktemp("dpq_plan")
    src, so = d / "plan.cpp", d / "plan.so"
    src.write_text(SHIM)
    subprocess.run([os.environ.get("CXX", "g++"), "-std=c++17", "-O2", "-fPIC", "-shared", "-I" + build.CSRC, "-o", str(so), str(src)],
                   check=True, capture_output=True)
    lib = ctypes.CDLL(str(so))

    def run(G, row_tiles, slots):
        out = (ctypes.c_int * (8 * G))()
        lib.steps(G, row_tiles, slots, out)
        return [[tuple(out[8 * b + 4 * i:8 * b + 4 * i + 4]) for i in range(2)] for b in range(G)]
    return run


@pytest.mark.parametrize("slots", [1, 8, 64, 296])
@pytest.mark.parametrize("row_tiles", [1, 2, 5, 32, 64, 224])
def test_every_task_follows_those_it_waits_for(steps, row_tiles, slots):
    depths = set()
    for G in list(range(1, 70)) + [112, 113, 131]:
        applied = [0] * G
        for b, trails in enumerate(steps(G, row_tiles, slots)):
            assert applied[b] == max(b - 1, 0)              # the block's own task adds the errors of block b - 1
            for errors, blocks, first, count in trails:
                for col in range(first, first + count):
                    assert b < col < G and applied[col] == errors and errors + blocks <= b
                    applied[col] += blocks
                    depths.add(blocks)
    assert depths == {1} if row_tiles * 130 < 2 * slots else max(depths) == 8 or row_tiles * 130 < 6 * slots
