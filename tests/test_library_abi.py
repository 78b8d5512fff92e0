"""Host-side checks that need no GPU: the C-ABI library builds, loads, and exports every symbol
include/keydiff.h declares; host-detectable errors are reported without any device work."""
import ctypes
import os
import re
import sysconfig

import pytest
import torch

from paper_2504_15364_b200 import binding, build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    build.build_library()
    return binding.load_library()


def test_header_symbols_are_exported(lib):
    header = open(os.path.join(ROOT, "include", "keydiff.h")).read()
    declared = set(re.findall(r"KEYDIFF_API\s+[\w\s\*]+?\b(keydiff_\w+)\s*\(", header))
    assert declared == set(binding.EXPORTS)
    for name in declared:
        assert hasattr(lib, name), name


def test_strerror_names_every_code(lib):
    texts = {lib.keydiff_strerror(c).decode() for c in range(0, -9, -1)}
    assert len(texts) == 9 and "unknown keydiff status" not in texts
    assert lib.keydiff_strerror(-99).decode() == "unknown keydiff status"


def test_null_and_bad_config_rejected_before_any_device_work(lib):
    out = ctypes.c_void_p()
    assert lib.keydiff_create(None, ctypes.byref(out)) == binding.KEYDIFF_ERR_INVALID_ARG
    cfg = binding.keydiff_config(1, 1, 8, 128, 512, 128, binding.KEYDIFF_BF16, 0, 0.0, 0)
    assert lib.keydiff_create(ctypes.byref(cfg), None) == binding.KEYDIFF_ERR_INVALID_ARG
    for field, bad in [("n_layers", 0), ("budget", 0), ("max_block", -1), ("device", -1), ("path", 7),
                       ("anchor_mode", 2), ("recent_window", -1), ("recent_window", 513), ("compaction", 2)]:
        c = binding.keydiff_config(1, 1, 8, 128, 512, 128, binding.KEYDIFF_BF16, 0, 0.0, 0)
        setattr(c, field, bad)
        assert lib.keydiff_create(ctypes.byref(c), ctypes.byref(out)) == binding.KEYDIFF_ERR_INVALID_ARG, field
    c = binding.keydiff_config(1, 1, 8, 64, 512, 128, binding.KEYDIFF_BF16, 0, 0.0, 0)      # head_dim 64
    assert lib.keydiff_create(ctypes.byref(c), ctypes.byref(out)) == binding.KEYDIFF_ERR_UNSUPPORTED
    c = binding.keydiff_config(1, 1, 8, 128, 512, 128, 5, 0, 0.0, 0)                          # dtype
    assert lib.keydiff_create(ctypes.byref(c), ctypes.byref(out)) == binding.KEYDIFF_ERR_UNSUPPORTED
    assert lib.keydiff_destroy(None) == binding.KEYDIFF_OK
    assert lib.keydiff_get_len(None, None) == binding.KEYDIFF_ERR_INVALID_ARG
    assert lib.keydiff_get_positions(None, None, None) == binding.KEYDIFF_ERR_INVALID_ARG
    assert lib.keydiff_evict(None, None, None, None, None, 1, 1, 1, 128, None) == binding.KEYDIFF_ERR_INVALID_ARG


def test_the_entry_of_evict_is_built_for_this_interpreter(lib):
    from paper_2504_15364_b200 import _pycall
    assert _pycall.__file__ == str(build.PYCALL) and build.PYCALL.name.endswith(sysconfig.get_config_var("EXT_SUFFIX"))
    assert not (build.PKG / "_pycall.so").exists() and binding._fast[0] is _pycall.evict


class FakeTensor:
    def __init__(self, numel, ptr, dtype=torch.bfloat16, is_cuda=True, contiguous=True):
        self.dtype, self.is_cuda, self._n, self._p, self._c = dtype, is_cuda, numel, ptr, contiguous

    numel = lambda self: self._n
    data_ptr = lambda self: self._p
    is_contiguous = lambda self: self._c


def test_the_entry_of_evict_without_its_c_module_is_the_same(lib):
    from paper_2504_15364_b200 import _pycall
    calls, status = [], [0]
    evict = binding._EVICT_TYPE(lambda *a: calls.append(a) or status[0])

    def get_len_of(ctx, out):
        out[0] = 77
        return 0
    get_len = binding._GET_LEN_TYPE(get_len_of)
    address = lambda f: ctypes.cast(f, ctypes.c_void_p).value
    row, budget = 256, 10
    good = [FakeTensor(budget * row, 16), FakeTensor(budget * row, 32), FakeTensor(3 * row, 48), FakeTensor(3 * row, 64)]
    cases = [(good, 0), (good, -5), ([good[0], good[1], good[2], FakeTensor(2 * row, 64)], 0), ([FakeTensor(9 * row, 16)] + good[1:], 0),
             (good[:2] + [FakeTensor(3 * row + 1, 48)] * 2, 0), (good[:3] + [FakeTensor(3 * row, 64, dtype=torch.float16)], 0),
             (good[:3] + [FakeTensor(3 * row, 64, is_cuda=False)], 0), ([FakeTensor(budget * row, 16, contiguous=False)] + good[1:], 0),
             (good[:2] + [FakeTensor(0, 0)] * 2, 0)]
    for tensors, rc in cases:
        status[0], seen = rc, []
        for entry in (_pycall.evict, binding._evict_ctypes):
            calls.clear()
            got = entry(address(evict), address(get_len), 1234, torch.bfloat16, budget, 2, 128, row, 99, *tensors)
            seen.append((got, list(calls)))
        assert seen[0] == seen[1], seen
    assert seen[0][1][0][6] == 0 and len(calls) == 1   # (an empty block is the library's to refuse)


@pytest.mark.skipif(torch.cuda.is_available(), reason="checks the no-GPU failure mode")
def test_create_fails_loudly_without_a_gpu(lib):
    # no CPU fallback: without a CUDA device the product path raises
    with pytest.raises(binding.KeyDiffError) as ei:
        binding.KeyDiff(1, 1, 8, 128, 512, 128)
    assert ei.value.code in (binding.KEYDIFF_ERR_CUDA, binding.KEYDIFF_ERR_UNSUPPORTED)
