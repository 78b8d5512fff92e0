"""The ordered layout on units that no cluster holds on chip (the launches on the running anchor), against the oracle.  Pinning
the cluster size to one block makes units of 1300 rows such units, so that the edges are reached at small sizes: blocks of one
row, blocks beyond the 1024 classes of the selection, ragged lengths, both variants, transition steps, equal scores."""
import numpy as np
import pytest
import torch

from oracle import compare
from paper_2504_15364_b200 import KeyDiff, binding, synth

pytestmark = pytest.mark.gpu


def bits(t):
    return t.detach().contiguous().view(torch.int16).cpu().numpy().view(np.uint16)


def check(kd, k, v, nk, nv, cur, N, **kw):
    pre_k, pre_v = bits(k), bits(v)
    kd.evict(k, v, nk, nv)
    torch.cuda.synchronize()
    sc = kd.scratch()
    assert int(sc["status"].item()) == 0
    compare.check_step(pre_k, pre_v, cur, bits(nk), bits(nv), N, bits(k), bits(v), sc["scores"].cpu().numpy(),
                       sc["kept_idx"].cpu().numpy(), n_threads=8, **kw)


@pytest.mark.parametrize("U,N,B,length,window,raw,model", [
    (3, 1300, 1, 1300, 0, 0, "outlier"), (2, 1531, 97, 1500, 33, 0, "drift"), (1, 2048, 1100, 2048, 0, 0, "offset"),
    (5, 1999, 640, 1999, 700, 1, "clusters"), (4, 4100, 129, 4100, 0, 1, "outlier"), (2, 3000, 1024, 2000, 0, 0, "clusters")])
def test_steps_match_the_oracle(monkeypatch, U, N, B, length, window, raw, model):
    monkeypatch.setenv("KEYDIFF_CLUSTER_SIZE", "1")
    wl = synth.Workload("t", 1, 1, U, 128, N, B, model, N + 5 * B, 71)
    k, v, stream = synth.prefilled_cache(wl, "cuda", length=length)
    kd = KeyDiff(1, 1, U, 128, N, B, anchor_mode=raw, recent_window=window)
    assert kd.launch_info()["path"] == binding.KEYDIFF_PATH_STAGED
    kd.set_len(length)
    for _ in range(4):
        cur = kd.len
        check(kd, k, v, *stream.next_block(B), cur, N, anchor_mode=raw, recent_window=window)
    kd.set_incremental(False)
    check(kd, k, v, *stream.next_block(B), N, N, anchor_mode=raw, recent_window=window)
    kd.close()


@pytest.mark.parametrize("U,N,B,length", [(2, 1300, 144, 1300), (1, 4096, 1, 4096), (3, 4111, 130, 4000), (16, 9000, 100, 9000)])
def test_units_moved_by_several_blocks(U, N, B, length):
    # two to eight blocks per unit and tensor, up to as many evicted rows as a block reads ahead; the last shape is dispatched
    # here by itself, and clustered keys evict rows all over the unit
    wl = synth.Workload("t", 1, 1, U, 128, N, B, "clusters", N + 4 * B, 72)
    k, v, stream = synth.prefilled_cache(wl, "cuda", length=length)
    with pytest.MonkeyPatch.context() as m:
        if N < 9000:
            m.setenv("KEYDIFF_CLUSTER_SIZE", "1")
        kd = KeyDiff(1, 1, U, 128, N, B)
    assert kd.launch_info()["path"] == binding.KEYDIFF_PATH_STAGED
    kd.set_len(length)
    for _ in range(3):
        cur = kd.len
        check(kd, k, v, *stream.next_block(B), cur, N)
    kd.close()


@pytest.mark.parametrize("U,N,at", [(16, 9000, 8000), (16, 9000, 8850), (3, 4111, 3300)])
def test_a_run_of_evicted_rows_near_the_end_moved_by_several_blocks(U, N, at):
    # as many rows go as a block reads ahead, and all behind them move by that much: eight short segments, whose sources lie as far
    # on as their direct successor's
    B = 144
    g = torch.Generator().manual_seed(N + at)
    k, v, nk, nv = (torch.randn(U, rows, 128, generator=g).to(torch.bfloat16) for rows in (N, N, B, B))
    run = torch.randn(U, 1, 128, generator=g) + 0.02 * torch.randn(U, B, 128, generator=g)   # one direction: the largest cosines
    k[:, at:at + B] = run.to(torch.bfloat16)
    k, v, nk, nv = k.cuda(), v.cuda(), nk.cuda(), nv.cuda()
    with pytest.MonkeyPatch.context() as m:
        if N < 9000:
            m.setenv("KEYDIFF_CLUSTER_SIZE", "1")
        kd = KeyDiff(1, 1, U, 128, N, B)
    assert kd.launch_info()["path"] == binding.KEYDIFF_PATH_STAGED
    kd.set_len(N)
    check(kd, k, v, nk, nv, N, N)
    assert torch.equal(kd.scratch()["first_evicted"].cpu(), torch.full((U,), at, dtype=torch.int32))
    kd.close()


def test_equal_scores_keep_the_older_token(monkeypatch):
    monkeypatch.setenv("KEYDIFF_CLUSTER_SIZE", "1")
    U, N, B = 2, 2500, 300
    g = torch.Generator().manual_seed(3)
    dirs = torch.randn(2, 128, generator=g)
    allk = dirs[torch.randint(0, 2, (U, N + 2 * B), generator=g)].to(torch.bfloat16).cuda()
    allv = torch.randn(U, N + 2 * B, 128, generator=g).to(torch.bfloat16).cuda()
    k, v = allk[:, :N].contiguous(), allv[:, :N].contiguous()
    kd = KeyDiff(1, 1, U, 128, N, B)
    kd.set_len(N)
    for s in range(2):
        sl = slice(N + s * B, N + (s + 1) * B)
        check(kd, k, v, allk[:, sl].contiguous(), allv[:, sl].contiguous(), N, N)
    kd.close()


@pytest.mark.parametrize("U,N,window,raw", [(185, 4099, 0, 0), (300, 2048, 17, 1)])
def test_single_evicted_rows_between_whole_blocks(U, N, window, raw):
    # units of the cluster kernel: steps that evict one row take the launches of this file, the anchor's sum passes from one
    # kind of step to the other and back; a step through the host entry brings the kept-index list
    wl = synth.Workload("t", 1, 1, U, 128, N, 128, "outlier", N + 8 * 128, 73)
    k, v, stream = synth.prefilled_cache(wl, "cuda", length=N)
    kd = KeyDiff(1, 1, U, 128, N, 128, anchor_mode=raw, recent_window=window)
    assert kd.launch_info()["path"] == binding.KEYDIFF_PATH_FUSED
    kd.set_len(N)
    for B in (128, 1, 1, 128, 96, 2, 128, 1):
        check(kd, k, v, *stream.next_block(B), N, N, anchor_mode=raw, recent_window=window)
    kept, status = torch.zeros(U, N, dtype=torch.int32).pin_memory(), torch.ones(1, dtype=torch.int32).pin_memory()
    nk, nv = (x.cpu().pin_memory() for x in stream.next_block(1))
    kd.evict_host(k, v, nk, nv, kept, status)
    torch.cuda.synchronize()
    assert int(status) == 0 and torch.equal(kept, kd.scratch()["kept_idx"].cpu())
    kd.close()


def test_a_captured_step_replayed_after_the_cache_was_refilled(monkeypatch):
    # a graph cannot know that appends or a restored cache made the carried sum stale: captured steps of these contexts carry none
    monkeypatch.setenv("KEYDIFF_CLUSTER_SIZE", "1")
    U, N, B = 2, 1400, 32
    wl = synth.Workload("t", 1, 1, U, 128, N, B, "drift", 3 * N, 75)
    k, v, stream = synth.prefilled_cache(wl, "cuda")
    kd = KeyDiff(1, 1, U, 128, N, B)
    assert kd.launch_info()["path"] == binding.KEYDIFF_PATH_STAGED
    kd.set_len(N)
    for _ in range(2):
        kd.evict(k, v, *stream.next_block(B))
    nk, nv = (x.clone() for x in stream.next_block(B))
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        kd.evict(k, v, nk, nv)
    kd.reset()
    while kd.len < N:   # another sequence
        kd.evict(k, v, *stream.next_block(min(B, N - kd.len)))
    for _ in range(3):
        for t, new in zip((nk, nv), stream.next_block(B)):
            t.copy_(new)
        pre_k, pre_v = bits(k), bits(v)
        g.replay()
        torch.cuda.synchronize()
        sc = kd.scratch()
        assert int(sc["status"].item()) == 0
        compare.check_step(pre_k, pre_v, N, bits(nk), bits(nv), N, bits(k), bits(v), sc["scores"].cpu().numpy(), sc["kept_idx"].cpu().numpy(),
                           n_threads=8)
    check(kd, k, v, *stream.next_block(B), N, N)   # and an eager step after them
    del g
    kd.close()


@pytest.mark.parametrize("U,N,B,slots,path,kernel", [
    (16, 9000, 100, 0, 0, "wide kernels (4 launches)"),   # could run in clusters of ten and is faster without
    (2, 20000, 64, 0, 0, "wide kernels (4 launches)"), (2, 700, 64, 0, 1, "staged kernels (4 launches)"), (2, 5000, 64, 0, 0, "fused_evict_kernel"),
    (8, 200, 20, 0, 0, "unit_evict_kernel"), (224, 2048, 128, 1, 0, "unit_evict_kernel"), (2, 5000, 64, 1, 0, "slot_evict_kernel")])
def test_launch_info_reports_what_runs(U, N, B, slots, path, kernel):
    kd = KeyDiff(1, 1, U, 128, N, B, path=path, compaction=slots)
    info = kd.launch_info()
    assert kd.kernel_name() == kernel
    if "4 launches" in kernel:
        assert info == {"path": binding.KEYDIFF_PATH_STAGED, "launches_per_step": 4, "cluster_size": 1}
    else:
        assert info["path"] == binding.KEYDIFF_PATH_FUSED and info["launches_per_step"] == 1
    kd.close()
