"""One thread block per unit (many small units, and long ones with slot reuse) against the oracle: the edges of the
all-at-once ranking (256 keys), of the selection's 1024 classes, of a tile and of the ring, both layouts and variants, transition
steps, blocks that are most of the unit, equal scores; and a second ctx on another stream at the same time."""
import numpy as np
import pytest
import torch

from oracle import compare
from paper_2504_15364_b200 import KeyDiff, binding, synth

pytestmark = pytest.mark.gpu


def bits(t):
    return t.detach().contiguous().view(torch.int16).cpu().numpy().view(np.uint16)


def run(U, N, B, length, slots, window=0, raw=0, model="outlier", steps=3, blocks=None, caches=None):
    wl = synth.Workload("t", 1, 1, U, 128, N, B, model, N + (steps + 1) * B, 83)
    if caches is None:
        k, v, stream = synth.prefilled_cache(wl, "cuda", length=length)
        blocks = [stream.next_block(B) for _ in range(steps)]
    else:
        k, v = caches
    kd = KeyDiff(1, 1, U, 128, N, B, anchor_mode=raw, recent_window=window, compaction=int(slots))
    info = kd.launch_info()
    assert info["path"] == binding.KEYDIFF_PATH_FUSED and info["cluster_size"] == 1
    kd.set_len(length)
    for step, (nk, nv) in enumerate(blocks):
        cur, pre_k, pre_v = kd.len, bits(k), bits(v)
        if slots:
            pos, nxt = kd.positions()
            torch.cuda.synchronize()
            pre_pos = np.tile(np.arange(N), (U, 1)) if step == 0 else pos.cpu().numpy().astype(np.int64)
        kd.evict(k, v, nk, nv)
        torch.cuda.synchronize()
        sc = kd.scratch()
        assert int(sc["status"].item()) == 0
        kw = dict(n_threads=8, anchor_mode=raw, recent_window=window)
        if slots:
            compare.check_step_slots(pre_k, pre_v, pre_pos, nxt, cur, bits(nk), bits(nv), N, bits(k), bits(v), sc["scores"].cpu().numpy(),
                                     sc["kept_idx"].cpu().numpy(), kd.positions()[0].cpu().numpy(), **kw)
        else:
            compare.check_step(pre_k, pre_v, cur, bits(nk), bits(nv), N, bits(k), bits(v), sc["scores"].cpu().numpy(),
                               sc["kept_idx"].cpu().numpy(), **kw)
    kd.close()


@pytest.mark.parametrize("slots", [False, True])
@pytest.mark.parametrize("U,N,B,length,window,raw,model", [
    (1, 1, 1, 1, 0, 0, "offset"), (3, 17, 16, 17, 5, 0, "outlier"), (90, 240, 16, 240, 0, 0, "drift"), (90, 240, 17, 240, 0, 1, "clusters"),
    (5, 130, 130, 100, 0, 0, "outlier"), (81, 500, 20, 490, 60, 0, "outlier"), (150, 700, 3, 700, 0, 1, "drift"),
    (100, 130, 390, 130, 0, 0, "clusters")])
def test_steps_match_the_oracle(slots, U, N, B, length, window, raw, model):
    run(U, N, B, length, slots, window, raw, model)


@pytest.mark.parametrize("U,N,B,length,window", [(60, 1000, 24, 1000, 300), (60, 1001, 99, 950, 0), (149, 1400, 100, 1400, 0),   # rows from global memory
                                                 (149, 1500, 1, 1500, 0), (150, 2040, 130, 2000, 0), (150, 1777, 1000, 1777, 900),   # the ring
                                                 (900, 4480, 33, 4480, 0)])
def test_long_units_with_slot_reuse(U, N, B, length, window):
    run(U, N, B, length, True, window, steps=2)


@pytest.mark.parametrize("slots", [False, True])
@pytest.mark.parametrize("N,B", [(200, 40), (460, 40)])
def test_equal_scores_keep_the_older_token(slots, N, B):
    U = 80
    g = torch.Generator().manual_seed(5)
    dirs = torch.randn(2, 128, generator=g)
    allk = dirs[torch.randint(0, 2, (U, N + 2 * B), generator=g)].to(torch.bfloat16).cuda()
    allv = torch.randn(U, N + 2 * B, 128, generator=g).to(torch.bfloat16).cuda()
    cut = lambda t, a, b: t[:, a:b].contiguous()
    run(U, N, B, N, slots, blocks=[(cut(allk, N + s * B, N + (s + 1) * B), cut(allv, N + s * B, N + (s + 1) * B)) for s in range(2)],
        caches=(cut(allk, 0, N), cut(allv, 0, N)))


@pytest.mark.parametrize("entry", ["ordered", "slots", "staged"])
@pytest.mark.parametrize("N,same,B", [(560, 300, 40), (700, 400, 40), (960, 900, 40), (640, 640, 300)])
def test_one_direction_repeated_crowds_the_list(entry, N, same, B):
    # more equal keys under the threshold than the selection's threshold bin may list, but not more than its list: the route that
    # passes from the list to the whole table
    U = 80
    g = torch.Generator().manual_seed(N)
    allk, allv = (torch.randn(U, N + 2 * B, 128, generator=g) for _ in range(2))
    allk[:, torch.randperm(N, generator=g)[:same]] = torch.randn(U, 1, 128, generator=g)
    allk, allv = allk.to(torch.bfloat16).cuda(), allv.to(torch.bfloat16).cuda()
    cut = lambda t, a, b: t[:, a:b].contiguous()
    blocks = [(cut(allk, N + s * B, N + (s + 1) * B), cut(allv, N + s * B, N + (s + 1) * B)) for s in range(2)]
    if entry != "staged":
        run(U, N, B, N, entry == "slots", blocks=blocks, caches=(cut(allk, 0, N), cut(allv, 0, N)))
        return
    k, v = cut(allk, 0, N), cut(allv, 0, N)
    static_k, static_v = k.clone(), v.clone()
    kd = KeyDiff(1, 1, U, 128, N, B, path=binding.KEYDIFF_PATH_STAGED)
    kd.set_len(N)
    for nk, nv in blocks:
        pre_k, pre_v = bits(k), bits(v)
        kd.evict(k, v, nk, nv)
        assert binding.evict_static(static_k, static_v, nk, nv, N) == N
        torch.cuda.synchronize()
        sc = kd.scratch()
        compare.check_step(pre_k, pre_v, N, bits(nk), bits(nv), N, bits(k), bits(v), sc["scores"].cpu().numpy(), sc["kept_idx"].cpu().numpy(),
                           n_threads=8)
        assert torch.equal(k, static_k) and torch.equal(v, static_v)
    kd.close()


def test_two_contexts_on_two_streams_do_not_disturb_each_other():
    wl = synth.Workload("t", 1, 1, 200, 128, 400, 40, "outlier", 400 + 10 * 40, 84)
    out = []
    for together in (False, True):
        got, work = [], []
        for slots in (0, 1):
            k, v, stream = synth.prefilled_cache(wl, "cuda")
            kd = KeyDiff(1, 1, 200, 128, 400, 40, compaction=slots)
            kd.set_len(400)
            work.append((kd, k, v, [stream.next_block(40) for _ in range(8)], torch.cuda.Stream()))
        torch.cuda.synchronize()
        for step in range(8):
            for kd, k, v, blocks, st in work:
                kd.evict(k, v, *blocks[step], stream=st)
                if not together:
                    torch.cuda.synchronize()
        torch.cuda.synchronize()
        for kd, k, v, _, _ in work:
            got += [k.clone(), v.clone(), kd.scratch()["kept_idx"].clone()]
            kd.close()
        out.append(got)
    assert all(torch.equal(a, b) for a, b in zip(*out))
