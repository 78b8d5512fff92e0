"""The block-wide selection (csrc/low_select.cuh) on the host: its own source, with threads as fibers (block_model.h), against a
sort.  Each warp in turn is held back as long as the others can run, so that a shared word that is written again
before every warp has read it changes the result or leaves threads waiting."""
import ctypes
import shutil
import subprocess
from pathlib import Path

import numpy as np
import pytest

TESTS = Path(__file__).resolve().parent
CSRC = TESTS.parent / "paper_2504_15364_b200" / "csrc"
BARRIER = r"""
#pragma once
#include "block_model.h"
namespace kd {
constexpr int kSelWarps = 8, kSelThreads = 256;
inline int sel_count(bool p) { model::block->f[model::block->self].pred = p; model::wait(model::kAtBarrier); return model::block->count; }
inline void sel_sync() { sel_count(false); }
}
"""
SOURCE = r"""
#include "block_model.h"
#include "low_select.cuh"
alignas(128) static kd::SelectorScratch scratch;
extern "C" int select_tokens(const uint32_t* keys, uint32_t* bitmap, uint32_t* work, int n, int E, int held_warp) {
    for (unsigned char* b = reinterpret_cast<unsigned char*>(&scratch); b < reinterpret_cast<unsigned char*>(&scratch + 1); ++b) *b = 0xa5;
    return model::run([&](int tid) { kd::Selector s(scratch, bitmap, work); kd::select_evicted(keys, n, E, tid, s); }, held_warp);
}
"""


@pytest.fixture(scope="module")
def select(tmp_path_factory):
    d = tmp_path_factory.mktemp("selection")
    shutil.copy(CSRC / "low_select.cuh", d)
    shutil.copy(TESTS / "block_model.h", d)
    bins = next(ln for ln in (CSRC / "fused_kernel.cuh").read_text().splitlines() if ln.startswith("constexpr int kBins ="))
    (d / "fused_kernel.cuh").write_text(f"#pragma once\nnamespace kd {{ {bins.split(';')[0]}; }}\n")
    (d / "sel_barrier.cuh").write_text(BARRIER)
    (d / "model.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-O1", "-std=c++17", "-Wno-unknown-pragmas", "-Wno-attributes", "-shared", "-fPIC", str(d / "model.cpp"), "-o",
                    str(d / "model.so")], check=True)
    lib = ctypes.CDLL(str(d / "model.so"))

    def call(keys, E, held_warp):
        n = len(keys)
        table = np.full((n + 3) // 4 * 4 + 16, 0xdeadbeef, np.uint32)
        at = (-table.ctypes.data // 4) % 4
        table[at:at + n] = keys
        bitmap, work = np.full((n + 31) // 32, 0x5a5a5a5a, np.uint32), np.full((n + 31) // 32, 0x5a5a5a5a, np.uint32)
        p = lambda a, o=0: ctypes.c_void_p(a.ctypes.data + 4 * o)
        assert lib.select_tokens(p(table, at), p(bitmap), p(work), n, E, held_warp) == 1, "threads wait for good"
        return np.flatnonzero(np.unpackbits(bitmap.view(np.uint8), bitorder="little"))

    return call


def tables(rng):
    wide = lambda n: rng.integers(0, 1 << 32, n, dtype=np.uint32)
    narrow = lambda n: (0x3f000000 + rng.integers(0, 1 << 20, n)).astype(np.uint32)
    for n, E in [(1, 1), (31, 7), (128, 128), (129, 3), (700, 40), (1023, 1023), (1500, 1100), (5000, 128)]:
        yield "spread", wide(n), E
        yield "close", narrow(n), E
    for n, same, E in [(700, 400, 40), (1000, 900, 300), (600, 300, 299), (640, 640, 128), (1900, 1500, 100), (3000, 3000, 1200)]:
        k = narrow(n)
        k[rng.permutation(n)[:same]] = 0x3effffff   # one direction repeated: more equal keys than the threshold bin may list
        yield "equal", k, E
    k = narrow(900)
    k[:500] = 0x3effffff
    k[500:760] = 0xffffffff   # a sliding window's tokens
    yield "window", k, 300
    yield "two keys", rng.choice(np.array([5, 0xffffff00], np.uint32), 800), 350


@pytest.mark.parametrize("held_warp", range(-1, 8))
def test_the_evicted_tokens_are_those_of_a_sort(select, held_warp):
    for name, keys, E in tables(np.random.default_rng(7)):
        n = len(keys)
        want = np.sort(np.lexsort((-np.arange(n), keys))[:E])   # key ascending, token descending
        assert np.array_equal(select(keys, E, held_warp), want), (name, n, E, held_warp)
