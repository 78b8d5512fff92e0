"""A step one of whose launches returns an error: the caller gets KEYDIFF_ERR_CUDA, the cache is as it was, and the step can be made again.
The launch is not made at all (a hook of the debug build, in a child process); nothing fails on the device."""
import os
import subprocess
import sys
import textwrap

import pytest

from paper_2504_15364_b200 import build

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = textwrap.dedent("""
    import ctypes, sys, torch
    from paper_2504_15364_b200 import binding, build, synth
    binding.LIB_PATH = build.DEBUG_LIB
    from paper_2504_15364_b200 import KeyDiff, KeyDiffError
    U, N, max_block, slots, _, *sizes = map(int, sys.argv[1:])
    wl = synth.Workload("t", 1, 1, U, 128, N, max_block, "drift", N + sum(sizes), 17)
    k0, v0, stream = synth.prefilled_cache(wl, "cuda")
    blocks = [stream.next_block(b) for b in sizes]
    fail_launch = binding.load_library().keydiff_debug_fail_launch
    fail_launch.argtypes = [ctypes.c_int32]
    read = binding.load_library().keydiff_debug_anchor_sum
    read.argtypes = [ctypes.c_void_p, ctypes.c_void_p]

    def run(nth):   # the last step's nth launch fails once (0: none does)
        k, v = k0.clone(), v0.clone()
        kd = KeyDiff(1, 1, U, 128, N, max_block, compaction=slots)
        kd.set_len(N)
        for b in blocks[:-1]:
            kd.evict(k, v, *b)
        torch.cuda.synchronize()
        failed = False
        if nth:
            before = k.clone(), v.clone()
            assert fail_launch(nth) == 0
            try:
                kd.evict(k, v, *blocks[-1])
            except KeyDiffError as e:
                assert e.code == binding.KEYDIFF_ERR_CUDA
                failed = True
            assert fail_launch(0) == 0
            torch.cuda.synchronize()
            assert not failed or (torch.equal(k, before[0]) and torch.equal(v, before[1])), "a failed step moved rows"
        if failed or not nth:
            kd.evict(k, v, *blocks[-1])
        total = torch.empty(U, 128, dtype=torch.float64)
        assert read(kd._ctx, total.data_ptr()) == 0 and int(kd.scratch()["status"].item()) == 0
        out = failed, total, k, v, kd.scratch()["kept_idx"].clone()
        kd.close()
        return out

    ref, launches = run(0), 0
    for nth in range(1, 9):
        got = run(nth)
        if not got[0]:
            break
        launches += 1
        print("CHANGE", nth, float((got[1] - ref[1]).abs().max()), all(torch.equal(a, b) for a, b in zip(got[2:], ref[2:])))
    print("LAUNCHES", launches)
""")


# units, budget, largest block, slot reuse, launches of the last step, sizes of the steps: several blocks per unit after a unit's block formed the sum,
# and where launches of their own did; units beyond a cluster; single rows of units that the cluster kernel serves otherwise; one block per
# unit; a cluster per unit
@pytest.mark.parametrize("args", [(150, 2000, 64, 1, 2, 64, 64, 1), (150, 4600, 33, 1, 2, 33, 33), (60, 10600, 50, 0, 4, 50, 50), (190, 2000, 40, 0, 4, 40, 40, 1),
                                  (90, 240, 17, 0, 1, 17, 17), (8, 4000, 33, 1, 1, 33, 33)])
def test_a_step_whose_launch_fails_can_be_made_again(args):
    build.build_library()
    build.build_library(debug_checks=True)
    r = subprocess.run([sys.executable, "-c", CHILD, *map(str, args)], capture_output=True, text=True, timeout=600, cwd=ROOT,
                       env={**os.environ, "PYTHONPATH": ROOT})
    assert r.returncode == 0, r.stderr[-2000:]
    lines = [ln.split() for ln in r.stdout.splitlines()]
    assert int(lines[-1][1]) == args[4], r.stdout
    for _, nth, change, same in lines[:-1]:
        # The sum is rebuilt where a launch may have changed it: of up to 2^14 terms of at most 1, in fp32 where launches of their own add
        # four rows at a time (2^-22 a row) or as the carried ones in double.  A block that is added twice changes it by its rows' terms.
        assert float(change) < 2.0 ** -8, r.stdout
        assert same == "True", r.stdout
