"""The list of evicted tokens (csrc/evicted_list.cuh) on the host: its own source, with threads as fibers (block_model.h); every list that the
block may hold, and a bitmap with more tokens than it has room for, as the debug build sees it."""
import ctypes
import shutil
import subprocess

import numpy as np
import pytest
from test_selection_model import BARRIER, CSRC, TESTS

COMMON = r"""
#pragma once
#include <cstdint>
#define KD_ROW_OK(d, limit, status) ((static_cast<unsigned>(d) < static_cast<unsigned>(limit)) || (*(status) = -8, false))
"""
SOURCE = r"""
#include "block_model.h"
#include "evicted_list.cuh"
alignas(128) static kd::SelectorScratch scratch;
extern "C" int list_tokens(uint32_t* bitmap, int* before, int* list, int n, int limit, int32_t* status, int* first, int held_warp) {
    return model::run([&](int tid) {
        kd::Selector s(scratch, bitmap, nullptr);
        const int f = kd::list_evicted(n, tid, s, before, list, limit, status);
        if (f != list[0]) *status = 1;
        *first = f;
    }, held_warp);
}
"""


@pytest.fixture(scope="module")
def list_evicted(tmp_path_factory):
    d = tmp_path_factory.mktemp("list")
    for name in ("low_select.cuh", "evicted_list.cuh"):
        shutil.copy(CSRC / name, d)
    shutil.copy(TESTS / "block_model.h", d)
    (d / "fused_kernel.cuh").write_text("#pragma once\nnamespace kd { constexpr int kBins = 2048; }\n")
    (d / "sel_barrier.cuh").write_text(BARRIER)
    (d / "common.cuh").write_text(COMMON)
    (d / "model.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-O1", "-std=c++17", "-Wno-unknown-pragmas", "-Wno-attributes", "-shared", "-fPIC", str(d / "model.cpp"), "-o",
                    str(d / "model.so")], check=True)
    lib = ctypes.CDLL(str(d / "model.so"))

    def call(n, tokens, limit, held_warp=-1):
        bits = np.zeros((n + 31) // 32 * 32, np.uint8)
        bits[tokens] = 1
        bitmap = np.packbits(bits, bitorder="little").view(np.uint32)
        before, out = np.full(len(bitmap), -1, np.int32), np.full(max(limit, len(tokens)) + 8, -1, np.int32)
        status, first = np.zeros(1, np.int32), np.zeros(1, np.int32)
        p = lambda a: ctypes.c_void_p(a.ctypes.data)
        assert lib.list_tokens(p(bitmap), p(before), p(out), n, limit, p(status), p(first), held_warp) == 1, "threads wait for good"
        words = np.add.reduceat(bits, np.arange(0, len(bits), 32), dtype=np.int32)
        return before, np.concatenate([[0], np.cumsum(words)[:-1]]), out, int(status[0]), int(first[0])

    return call


@pytest.mark.parametrize("held_warp", [-1, 0, 3, 7])
@pytest.mark.parametrize("n,E", [(1, 1), (32, 32), (33, 1), (700, 64), (8192, 128), (8320, 128), (8193, 1024), (20001, 640)])
def test_the_list_is_the_bitmap(list_evicted, n, E, held_warp):
    tokens = np.sort(np.random.default_rng(n).permutation(n)[:E])
    before, want_before, out, status, first = list_evicted(n, tokens, E, held_warp)
    assert status == 0 and first == tokens[0]
    assert np.array_equal(out[:E], tokens) and (out[E:] == -1).all() and np.array_equal(before, want_before)


@pytest.mark.parametrize("n,E,limit", [(700, 64, 63), (8320, 129, 128), (8320, 8320, 128)])
def test_tokens_beyond_the_room_are_reported_and_not_written(list_evicted, n, E, limit):
    tokens = np.sort(np.random.default_rng(n).permutation(n)[:E])
    _, _, out, status, _ = list_evicted(n, tokens, limit)
    assert status == -8 and np.array_equal(out[:limit], tokens[:limit]) and (out[limit:] == -1).all()
