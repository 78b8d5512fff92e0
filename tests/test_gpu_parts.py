"""Slot reuse with several blocks per unit (csrc/parts_kernel.cuh) against the oracle: ragged parts, both variants, transition steps, blocks of one row,
either way to the first sum, host entry and capture; which kernel serves which shape and step, and what the others give for the same steps."""
import pytest
import torch

from paper_2504_15364_b200 import KeyDiff, binding, synth
from test_gpu_row_edges import check_steps

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("U,N,length,blocks,window,raw,model", [
    (150, 2000, 2000, (128, 128, 1), 0, 0, "outlier"),            # a block per unit forms the first sum; 2128 = 4 parts of 512 and 80 rows
    (177, 2047, 2000, (130, 130, 7), 400, 0, "clusters"),         # the first step also fills empty slots; single keys, window beyond the block
    (160, 2304, 2304, (1, 256, 1, 255), 20, 1, "drift"),
    (450, 1999, 1999, (3, 3), 0, 0, "offset"),
    (150, 2001, 2001, (40, 9, 40), 1500, 1, "clusters"),          # windows far beyond a block, positions out of order
    (300, 4601, 4601, (33, 33), 4600, 0, "drift"),
    (150, 4600, 4600, (33, 33, 1), 0, 0, "outlier"),              # the first sum comes from launches of its own
    (149, 10200, 10200, (64, 64), 0, 0, "drift"),                 # two blocks per SM, though three would fit
    (149, 13000, 13000, (64, 64), 0, 0, "outlier"),               # two fit
    (450, 1950, 1950, (1023, 1, 1023), 0, 0, "offset"),           # three lists of blocks this large take more than the keys
    (150, 3900, 3900, (700, 5, 700), 900, 0, "outlier")])
def test_steps_match_the_oracle(U, N, length, blocks, window, raw, model):
    check_steps(U, N, max(blocks), length, True, model=model, kernel="parts_kernel", blocks=blocks, recent_window=window, anchor_mode=raw)


def steps_of(path, k0, v0, blocks, window, incremental=True, reset_at=None):
    """What the steps leave, from a copy of a full cache; with reset_at the step of that number is the first of a new sequence over the same rows."""
    U, N = k0.shape[0], k0.shape[1]
    k, v = k0.clone(), v0.clone()
    kd = KeyDiff(1, 1, U, 128, N, max(b[0].shape[-2] for b in blocks), path=path, recent_window=window, compaction=binding.KEYDIFF_COMPACT_SLOT_REUSE)
    kd.set_incremental(incremental)
    kd.set_len(N)
    scores = []
    for i, b in enumerate(blocks):
        if i == reset_at:
            kd.reset()
            kd.set_len(N)
        kd.evict(k, v, *b)
        scores.append(kd.scratch()["scores"].clone())
    torch.cuda.synchronize()
    assert int(kd.scratch()["status"].item()) == 0
    out = k, v, kd.positions()[0].clone(), kd.scratch()["kept_idx"].clone(), torch.stack(scores)
    name = kd.kernel_name()
    kd.close()
    return name, out


@pytest.mark.parametrize("U,N,B,window,incremental,reset_at", [(150, 2000, 64, 0, True, None), (450, 2047, 100, 600, True, None), (150, 2000, 64, 300, True, 2),
                                                               (150, 2000, 64, 0, False, None), (150, 4600, 33, 0, True, None), (300, 4500, 64, 1000, True, 2),
                                                               (150, 4600, 33, 0, False, 1)])
def test_the_kernels_that_serve_these_shapes_with_the_fused_path_agree(U, N, B, window, incremental, reset_at):
    wl = synth.Workload("t", 1, 1, U, 128, N, B, "drift", N + 5 * B, 93)
    k0, v0, stream = synth.prefilled_cache(wl, "cuda")
    blocks = [stream.next_block(b) for b in (B, B, 1, B)]
    name, out = steps_of(binding.KEYDIFF_PATH_AUTO, k0, v0, blocks, window, incremental, reset_at)
    old, ref = steps_of(binding.KEYDIFF_PATH_FUSED, k0, v0, blocks, window, incremental, reset_at)
    assert name == ("parts_kernel" if incremental or N > 4400 else "unit_evict_kernel") and old == ("unit_evict_kernel" if N < 4400 else "slot_evict_kernel")
    if old == "unit_evict_kernel":   # the same additions in the same order
        assert all(torch.equal(a, b) for a, b in zip(out, ref))
        return
    # A unit's cluster adds the same terms in another order (block rows and evicted ones together): sums in double, an anchor that may round
    # the other way in fp32, 2^-24 of it, and with it the scores: 128 products, 2^-24 each at most of |mu| |k|.
    assert all(torch.equal(a, b) for a, b in zip(out[:4], ref[:4]))
    assert float((out[4] - ref[4]).abs().max()) <= 2.0 ** -24 * 128


@pytest.mark.parametrize("U,N,blocks,window", [(160, 2500, (600, 1, 600, 64, 512, 513), 0), (640, 1950, (384, 16, 384, 1), 500)])
def test_a_block_per_unit_takes_the_large_blocks_of_a_context(U, N, blocks, window):
    check_steps(U, N, max(blocks), N, True, model="offset", kernel="unit_evict_kernel", blocks=blocks, recent_window=window)


@pytest.mark.parametrize("U,N,B,kernel", [(148, 2048, 128, "slot_evict_kernel"), (178, 2048, 128, "unit_evict_kernel"), (150, 1900, 64, "unit_evict_kernel"),
                                          (237, 8192, 128, "slot_evict_kernel"), (236, 8192, 128, "parts_kernel"), (297, 8192, 128, "parts_kernel"),
                                          (110, 12000, 64, "slot_evict_kernel"), (400, 12000, 64, "slot_evict_kernel"), (445, 2048, 64, "parts_kernel"),
                                          # large blocks, and where parts leave an SM no L1 or only two blocks: 3 to 15 % slower with several per unit
                                          (149, 2048, 1024, "unit_evict_kernel"), (177, 2300, 512, "unit_evict_kernel"), (683, 1900, 384, "unit_evict_kernel"),
                                          (600, 2048, 256, "parts_kernel"), (1000, 8192, 1024, "parts_kernel"), (400, 8192, 512, "parts_kernel"),
                                          (400, 9700, 64, "parts_kernel"), (400, 9900, 256, "slot_evict_kernel"), (236, 9900, 256, "slot_evict_kernel"),
                                          (400, 9900, 640, "parts_kernel"), (1000, 9900, 256, "unit_evict_kernel"), (330, 10156, 128, "parts_kernel"),
                                          (200, 12000, 64, "slot_evict_kernel"), (190, 12000, 640, "parts_kernel"), (190, 18000, 16, "slot_evict_kernel"),
                                          (177, 20000, 16, "parts_kernel"), (330, 18000, 16, "slot_evict_kernel"),
                                          (236, 4650, 200, "slot_evict_kernel"), (222, 4650, 200, "parts_kernel"), (400, 6100, 200, "slot_evict_kernel"),
                                          (1025, 9500, 640, "unit_evict_kernel"), (177, 3100, 256, "parts_kernel"), (149, 1910, 128, "unit_evict_kernel")])
def test_which_kernel_serves(U, N, B, kernel):
    kd = KeyDiff(1, 1, U, 128, N, B, compaction=binding.KEYDIFF_COMPACT_SLOT_REUSE)
    assert kd.kernel_name() == kernel
    info = kd.launch_info()
    assert info["path"] == binding.KEYDIFF_PATH_FUSED and info["launches_per_step"] == (2 if kernel == "parts_kernel" else 1)
    kd.close()


@pytest.mark.parametrize("U,N,B,carried,rebuilt", [(150, 2048, 64, "parts_kernel", "unit_evict_kernel"), (1000, 8192, 64, "parts_kernel", "unit_evict_kernel"),
                                                    (150, 8192, 64, "parts_kernel", "parts_kernel"), (177, 2300, 512, "unit_evict_kernel", "unit_evict_kernel")])
def test_the_facts_reported_are_those_of_a_step_as_the_context_stands(U, N, B, carried, rebuilt):
    kd = KeyDiff(1, 1, U, 128, N, B, compaction=binding.KEYDIFF_COMPACT_SLOT_REUSE)
    for on, kernel in ((True, carried), (False, rebuilt), (True, carried)):
        kd.set_incremental(on)
        assert kd.kernel_name() == kernel and kd.launch_info()["launches_per_step"] == (2 if kernel == "parts_kernel" else 1)
    kd.close()


@pytest.mark.parametrize("N", [2000, 4600])
def test_captured_steps_and_the_host_entry_give_the_same(N):
    U, B = 150, 64
    wl = synth.Workload("t", 1, 1, U, 128, N, B, "outlier", N + 8 * B, 92)
    k0, v0, stream = synth.prefilled_cache(wl, "cuda")
    blocks = [stream.next_block(B) for _ in range(5)]
    out = []
    for way in ("eager", "captured", "host"):
        k, v = k0.clone(), v0.clone()
        kd = KeyDiff(1, 1, U, 128, N, B, compaction=binding.KEYDIFF_COMPACT_SLOT_REUSE)
        kd.set_len(N)
        kept = kd.scratch()["kept_idx"]
        if way == "host":
            kept, status = torch.zeros(U, N, dtype=torch.int32).pin_memory(), torch.ones(1, dtype=torch.int32).pin_memory()
            for nk, nv in blocks:
                kd.evict_host(k, v, nk.cpu().pin_memory(), nv.cpu().pin_memory(), kept, status)
                torch.cuda.synchronize()
            assert int(status) == 0
        else:
            kd.evict(k, v, *blocks[0])
            torch.cuda.synchronize()
            g = torch.cuda.CUDAGraph()
            if way == "captured":
                with torch.cuda.graph(g):
                    for b in blocks[1:]:
                        kd.evict(k, v, *b)
                g.replay()
            else:
                for b in blocks[1:]:
                    kd.evict(k, v, *b)
            torch.cuda.synchronize()
            del g
        assert int(kd.scratch()["status"].item()) == 0
        out.append([k, v, kept.cpu().clone(), kd.positions()[0].clone()])
        kd.close()
    for other in out[1:]:
        assert all(torch.equal(a, b) for a, b in zip(out[0], other))
