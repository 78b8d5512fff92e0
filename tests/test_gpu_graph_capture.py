"""Steps captured into a CUDA graph give the bits of the same steps launched eagerly: appends, the transition to a full
cache and evicting steps, whose kernels are chained by programmatic dependent launches, on every path and layout."""
import pytest
import torch

from paper_2504_15364_b200 import KeyDiff, binding, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("slots", [False, True])
@pytest.mark.parametrize("path", [binding.KEYDIFF_PATH_STAGED, binding.KEYDIFF_PATH_FUSED])
@pytest.mark.parametrize("U,N,B", [(3, 512, 128), (9, 777, 50)])
def test_captured_steps_match_eager_steps(U, N, B, path, slots):
    wl = synth.Workload("t", 1, 1, U, 128, N, B, "outlier", 4 * N, 61)
    out = []
    for captured in (False, True):
        stream = synth.KVStream(wl, "cuda")
        k = torch.zeros(U, N, 128, dtype=torch.bfloat16, device="cuda")
        v = torch.zeros_like(k)
        kd = KeyDiff(1, 1, U, 128, N, B, path=path, compaction=int(slots))
        blocks = [stream.next_block(B) for _ in range(N // B + 4)]
        for b in blocks[:2]:
            kd.evict(k, v, *b)
        torch.cuda.synchronize()
        if captured:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g):
                for b in blocks[2:]:
                    kd.evict(k, v, *b)
            g.replay()
        else:
            for b in blocks[2:]:
                kd.evict(k, v, *b)
        torch.cuda.synchronize()
        assert kd.len == N and int(kd.scratch()["status"].item()) == 0
        out.append([k, v, kd.scratch()["kept_idx"].clone()] + ([kd.positions()[0].clone()] if slots else []))
        if captured:
            del g
        kd.close()
    assert all(torch.equal(a, b) for a, b in zip(*out))


@pytest.mark.parametrize("sizes", [(64, 1), (1, 64), (1, 1), (1, 64, 1, 1)])
def test_replayed_steps_go_on_like_eager_ones(sizes):
    # units of the cluster kernel whose single evicted rows take four launches: an even number of steps, captured once and replayed,
    # carries the anchor's sum on from replay to replay, whichever kind the steps are
    U, N = 185, 2048
    wl = synth.Workload("t", 1, 1, U, 128, N, 64, "outlier", N + 4 * 64, 62)
    k0, v0, stream = synth.prefilled_cache(wl, "cuda")
    start, blocks = [stream.next_block(b) for b in (64, 1, 64)], [stream.next_block(b) for b in sizes]
    out = []
    for captured in (False, True):
        k, v = k0.clone(), v0.clone()
        kd = KeyDiff(1, 1, U, 128, N, 64)
        kd.set_len(N)
        for b in start:
            kd.evict(k, v, *b)
        torch.cuda.synchronize()
        if captured:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g):
                for b in blocks:
                    kd.evict(k, v, *b)
            for _ in range(3):
                g.replay()
        else:
            for b in blocks * 3:
                kd.evict(k, v, *b)
        torch.cuda.synchronize()
        assert int(kd.scratch()["status"].item()) == 0
        out.append([k, v, kd.scratch()["kept_idx"].clone(), kd.scratch()["scores"][:, :N + sizes[-1]].clone()])
        if captured:
            del g
        kd.close()
    assert all(torch.equal(a, b) for a, b in zip(*out))
