"""Tuned choices are kept per alignment of the planes: what was timed on aligned
ones is not replayed on others; pins and caches without the alignment hold for
both.  (The CPU part goes through the cache file; the GPU part times.)"""
import json

import pytest

from paper_2504_01266_gb300 import _lib as L


@pytest.fixture()
def lib():
    from paper_2504_01266_gb300 import build
    build.build()
    mode = L.giga_autotune_get_mode()
    L.giga_autotune_clear()
    L.giga_autotune_set_mode(1)
    yield L
    L.giga_autotune_clear()
    L.giga_autotune_set_mode(mode)


def desc(W, dtype=0):
    return L.desc(1, 1, 1, 1024, W, 3, 1, 0, dtype, L.GIGA_LAYOUT_NCHW)


def load(path, entries):
    path.write_text(json.dumps({"giga_autotune": 1, "entries": entries}))
    assert L.giga_autotune_load(str(path)) == L.GIGA_OK


def choices(op=1):
    """Of an aligned and an unaligned problem in the same size class."""
    return L.giga_autotune_choice(desc(1024), op), L.giga_autotune_choice(desc(1025), op)


def test_cache_keys(lib, tmp_path):
    path = tmp_path / "cache.json"
    load(path, {"0:0:3:0:20:0": 2})
    assert choices() == (2, 0)
    load(path, {"0:0:3:0:20:1": 5})
    assert choices() == (2, 5)
    # BF16: W = 1028 allows 8-byte accesses, not TMA
    load(path, {"0:1:3:0:20:0": 4})
    assert L.giga_autotune_choice(desc(1032, 1), 1) == 4
    assert L.giga_autotune_choice(desc(1028, 1), 1) == 0
    # without the alignment: both, in place of what was there
    load(path, {"0:0:3:0:20": 3})
    assert choices() == (3, 3)
    # a pin too; a file keeps all three kinds
    load(path, {"0:0:3:0:20:1": 6})
    assert choices() == (3, 6)
    assert L.giga_autotune_save(str(path)) == L.GIGA_OK
    L.giga_autotune_clear()
    assert L.giga_autotune_load(str(path)) == L.GIGA_OK and choices() == (3, 6)
    assert L.giga_autotune_set_choice(desc(1025), 1, 7) == L.GIGA_OK
    assert choices() == (7, 7)


@pytest.mark.gpu
def test_tuning_one_alignment_leaves_the_other(lib, tmp_path):
    import torch
    path = str(tmp_path / "tuned.json")
    stream = torch.cuda.current_stream().cuda_stream
    for count, W in ((1, 1024), (2, 1025)):
        x = torch.rand((1, 1, 1024, W), device="cuda")
        y, w = torch.empty_like(x), torch.rand((1, 3, 3), device="cuda")
        L.check(L.giga_autotune_conv2d(desc(W), 1, x.data_ptr(), w.data_ptr(), y.data_ptr(), 0, 0,
                                       0, 0, 0, stream), "autotune")
        assert L.giga_autotune_save(path) == L.GIGA_OK
        entries = json.load(open(path))["entries"]
        assert len(entries) == count, entries
