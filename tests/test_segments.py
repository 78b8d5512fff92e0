"""How a unit's rows are split over the blocks that move them (csrc/segments.h, compiled for the host): a block waits only for
the block in front of it, so what it reads beyond its own rows must lie in the rows of its direct successor."""
import ctypes
import subprocess
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parent.parent / "paper_2504_15364_b200" / "csrc"
SOURCE = r"""
#include "segments.h"
#include <vector>
using namespace kd;
// A unit of N cached and E new rows that evicts rows [at, at + E): the rows that a segment reads ahead from beyond its direct successor,
// or not ahead from beyond its own end, and the segments that do not join up or read too many rows ahead.
static int misplaced(int N, int E, int at, int segments) {
    int bad = 0;
    auto source = [&](int d) { return d < at ? d : d + E; };
    for (int s = 0; s < segments; ++s) {
        const Segment g = segment_of(at, N, segments, s);
        if (s > 0 && g.d0 != segment_of(at, N, segments, s - 1).d1) ++bad;
        if (g.d0 == g.d1) continue;
        const int m = rows_read_ahead(g, N, source(g.d1 - 1)), successor_end = segment_of(at, N, segments, s + 1).d1;
        bad += m < 0 || m > kHaloRows || m > g.d1 - g.d0;
        for (int d = g.d0; d < g.d1; ++d) {
            const int from = source(d);
            if (from >= N) continue;   // a block row: nobody writes it
            bad += from >= (d >= g.d1 - m ? (g.d1 < N ? successor_end : N) : g.d1);
        }
    }
    return bad + (segment_of(at, N, segments, segments - 1).d1 != N);
}
// ... for every run that begins in [from, N]
extern "C" int misplaced_reads(int N, int E, int from, int segments) {
    int bad = 0;
    for (int at = from; at <= N; ++at) bad += misplaced(N, E, at, segments);
    return bad;
}
"""


@pytest.fixture(scope="module")
def model(tmp_path_factory):
    d = tmp_path_factory.mktemp("segments")
    (d / "model.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", f"-I{CSRC}", str(d / "model.cpp"), "-o", str(d / "model.so")], check=True)
    return ctypes.CDLL(str(d / "model.so")).misplaced_reads


@pytest.mark.parametrize("segments", range(2, 9))
def test_a_segment_reads_no_further_than_its_direct_successor(model, segments):
    N = 512 * segments + 37
    for E in (1, 100, 128, 129, 136, 144):
        assert model(N, E, 0, segments) == 0, (segments, E)


def test_a_run_of_evicted_rows_near_the_end_of_a_long_unit(model):
    assert model(9000, 144, 6000, 8) == 0
