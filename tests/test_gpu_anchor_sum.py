"""The anchor's running sum does not drift, whichever kernels serve the steps.  With a sliding window of N tokens the oldest ones go;
a stream that repeats itself every P > N tokens then leaves the same rows in the cache after P tokens, and the sum must be what it was:
every row takes away the very terms that it brought.  The sum is read through the debug build, in a child process."""
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
    from paper_2504_15364_b200 import binding, build
    binding.LIB_PATH = build.DEBUG_LIB
    from paper_2504_15364_b200 import KeyDiff
    U, N, P, slots, raw, *pattern = map(int, sys.argv[1:])
    g = torch.Generator(device="cuda").manual_seed(N)
    rows = (torch.randn(U, P, 128, generator=g, device="cuda") * 3).to(torch.bfloat16)
    k = rows[:, :N].contiguous()
    v = k.clone()
    kd = KeyDiff(1, 1, U, 128, N, max(pattern), anchor_mode=raw, recent_window=N, compaction=slots)
    kd.set_len(N)
    read = binding.load_library().keydiff_debug_anchor_sum
    read.argtypes = [ctypes.c_void_p, ctypes.c_void_p]
    def total():
        out = torch.empty(U, 128, dtype=torch.float64)
        assert read(kd._ctx, out.data_ptr()) == 0
        return out
    at = N
    def turn():
        global at
        for B in pattern:
            block = rows[:, (torch.arange(at, at + B, device="cuda") % P)].contiguous()
            kd.evict(k, v, block, block)
            at += B
    def held():   # which rows the cache holds, by their first eight bytes
        return torch.sort(k.view(torch.int64).view(U, N, 32)[:, :, 0], 1).values
    turn()   # (the first step rebuilds the sum from all rows)
    start, first, rows_then = at, total(), held()
    while at < start + 2 * P:
        turn()
    assert (at - start) % P == 0 and int(kd.scratch()["status"].item()) == 0
    assert torch.equal(held(), rows_then), "the stream did not leave the same rows"
    print("LARGEST CHANGE", float((total() - first).abs().max()))
    kd.close()
""")


# steps of the cluster kernel and single rows through the four launches (what came in a block goes by itself and the other way round:
# N is three and a half turns); the same on the raw anchor; the four launches alone; one block per unit; slot reuse, one block and clusters;
# several blocks per unit, their steps in turn with a block per unit's (which rebuilds the sum every 1024 steps, and takes the large blocks)
@pytest.mark.parametrize("args,cluster", [((185, 2100, 2400, 0, 0, 500) + (1,) * 100, 0), ((300, 2048, 2072, 0, 1, 33, 1, 1, 2), 0),
                                          ((3, 1500, 1656, 0, 0, 97, 1, 40), 1), ((90, 240, 276, 0, 0, 16, 7), 0),
                                          ((8, 500, 606, 1, 0, 100, 1), 0), ((8, 4000, 4128, 1, 0, 128, 1), 0),
                                          ((150, 4600, 4692, 1, 0, 64, 5), 0), ((150, 2000, 2100, 1, 0, 100) + (1,) * 600, 0),
                                          ((150, 2400, 2756, 1, 1, 600, 64, 20, 5), 0)])
def test_the_sum_is_unchanged_when_the_rows_are(args, cluster):
    build.build_library()
    build.build_library(debug_checks=True)
    env = {**os.environ, "PYTHONPATH": ROOT}
    if cluster:
        env["KEYDIFF_CLUSTER_SIZE"] = str(cluster)
    r = subprocess.run([sys.executable, "-c", CHILD, *map(str, args)], capture_output=True, text=True, timeout=600, cwd=ROOT, env=env)
    assert r.returncode == 0, r.stderr[-2000:]
    change = float(r.stdout.split("LARGEST CHANGE")[1])
    # Terms of at most 1 (raw anchor: 2^5), block sums under 2^9, the running sum under 2^12.  Per channel at most 2^14 additions to block
    # sums, which round by 2^-44 each, and 2^14 to the running sum, 2^-41 each: less than 2^-26 together, and 0 is seen.  One
    # term that goes as another than it came leaves up to 2^-25, and hundreds of them add up (1.3e-6 when the two kinds of step had two forms).
    assert change < 2.0 ** -26 * (2 ** 5 if args[4] else 1), change
