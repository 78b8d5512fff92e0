"""Steps of the block per unit at the row counts where its inner loops change: how many rows' terms are requested together (steps of 16
rows, up to four), against the oracle."""
import numpy as np
import pytest
import torch

from oracle import compare
from paper_2504_15364_b200 import KeyDiff, synth

pytestmark = pytest.mark.gpu


def bits(t):
    return t.detach().contiguous().view(torch.int16).cpu().numpy().view(np.uint16)


def check_steps(U, N, B, length, slots, steps=3, model="outlier", kernel=None, blocks=None, **kw):
    """`steps` steps of B rows (or those of `blocks`) from a cache of `length` rows, each against the oracle."""
    sizes = blocks or [B] * steps
    wl = synth.Workload("t", 1, 1, U, 128, N, B, model, N + sum(sizes) + B, 91)
    k, v, stream = synth.prefilled_cache(wl, "cuda", length=length)
    raw, window = kw.get("anchor_mode", 0), kw.get("recent_window", 0)
    kd = KeyDiff(1, 1, U, 128, N, B, anchor_mode=raw, recent_window=window, compaction=int(slots))
    assert kernel is None or kd.kernel_name() == kernel
    kd.set_len(length)
    for step, b in enumerate(sizes):
        nk, nv = stream.next_block(b)
        cur, pre_k, pre_v = kd.len, bits(k), bits(v)
        if slots:
            pos, nxt = kd.positions()
            torch.cuda.synchronize()
            pre_pos = np.tile(np.arange(N), (U, 1)) if step == 0 else pos.cpu().numpy().astype(np.int64)
        kd.evict(k, v, nk, nv)
        torch.cuda.synchronize()
        sc = kd.scratch()
        assert int(sc["status"].item()) == 0
        args = (cur, bits(nk), bits(nv), N, bits(k), bits(v), sc["scores"].cpu().numpy(), sc["kept_idx"].cpu().numpy())
        if slots:
            compare.check_step_slots(pre_k, pre_v, pre_pos, nxt, *args, kd.positions()[0].cpu().numpy(), n_threads=8, **kw)
        else:
            compare.check_step(pre_k, pre_v, *args, n_threads=8, **kw)
    kd.close()


@pytest.mark.parametrize("slots", [False, True])
@pytest.mark.parametrize("B", [1, 2, 15, 16, 17, 32, 33, 48, 49, 64, 65, 100])
def test_rows_around_the_depths_of_the_terms(B, slots):
    check_steps(5, 130, B, 130, slots, kernel="unit_evict_kernel")


@pytest.mark.parametrize("B", [16, 17, 32, 33, 64, 65, 80, 81, 128, 129, 144, 193, 257])
def test_rows_around_the_depths_of_the_long_units_terms(monkeypatch, B):
    monkeypatch.setenv("KEYDIFF_CLUSTER_SIZE", "1")   # units of this size then take the launches for long units: up to eight rows together
    check_steps(2, 1500, B, 1500, False, kernel="wide kernels (4 launches)", model="drift")


@pytest.mark.parametrize("N,length", [(640, 640), (641, 641), (640, 636), (640, 637), (643, 640), (12, 4), (9, 1)])
def test_slot_lists_written_four_entries_at_a_time_or_not(N, length):
    check_steps(3, N, 9, length, True)   # (more rows than there are empty slots: every step evicts)


@pytest.mark.parametrize("N,B,window", [(1301, 131, 0), (1300, 131, 40), (1298, 2, 7), (1300, 4, 1300 - 3)])
def test_scores_read_four_at_a_time_or_not(monkeypatch, N, B, window):
    monkeypatch.setenv("KEYDIFF_CLUSTER_SIZE", "1")   # units of this size then take the launches for long units
    check_steps(2, N, B, N, False, blocks=[B, B, max(B - 1, 1)], kernel="wide kernels (4 launches)", recent_window=window)
