"""Which body a batch runs with (no GPU): an unroll that was set is the one that
is run, the built-in one follows the batch, and the cache file keeps which of the
two a bucket has."""
import json

import numpy as np
import pytest

import paper_1309_1894_gb300 as wx
from paper_1309_1894_gb300 import binding

vectors = binding.wxpy_debug_batch_vectors
B = 0x7F0000000000


@pytest.fixture(autouse=True)
def reset():
    wx.wxpy_batch_shape_reset()
    yield
    wx.wxpy_batch_shape_reset()
    wx.wxpy_tune_clear()


def table(ns):
    ns = np.asarray(ns, np.int64)
    at = B + 32 * np.concatenate([[0], np.cumsum((ns + 3) // 4)[:-1]])
    return wx.desc_table(ns, np.ones(len(ns)), *(at + (k << 40) for k in range(3)))


SHORT = table([900] * 9000)          # tiles of 900 elements (bucket 9)
LONG = table([1 << 16] * 1000)       # tiles of 8192 (bucket 16)
MIXED = table([900] * 9000 + [1 << 16] * 1000)


def test_the_built_in_unroll_follows_the_batch():
    assert wx.wxpy_batch_shape_get(9) == (0, 4)  # as it is reported
    assert vectors(SHORT) == 2 and vectors(LONG) == 4 and vectors(MIXED) == 4
    assert vectors(table([0, 0])) == 2


def test_an_unroll_that_was_set_is_run():
    wx.wxpy_batch_shape_set(9, 0, 4)
    assert vectors(SHORT) == 4
    wx.wxpy_batch_shape_set(9, 0, 2)
    assert vectors(SHORT) == 2 and vectors(MIXED) == 4
    wx.wxpy_batch_shape_set(16, 8192, 2)
    assert vectors(LONG) == 2 and vectors(MIXED) == 2
    wx.wxpy_batch_shape_set(16, 8192, 4)
    assert vectors(LONG) == 4 and vectors(SHORT) == 2
    wx.wxpy_batch_shape_set(9, 0, 4)
    wx.wxpy_batch_shape_set(16, 8192, 1)
    assert vectors(MIXED) == 4 and vectors(LONG) == 2


@pytest.mark.parametrize("built_in,want", [(None, 4), (0, 4), (1, 2)])
def test_a_cache_file_keeps_which_it_was(tmp_path, built_in, want):
    entry = {"bucket": 9, "tile": 0, "unroll_log2": 2}
    if built_in is not None:
        entry["built_in"] = built_in
    p = tmp_path / "c.json"
    doc = {"format": "wxpy-tune-1", "device": "X", "batch": [entry], "entries": []}
    p.write_text(json.dumps(doc))
    wx.wxpy_tune_cache_load(str(p), check_device=False)
    assert vectors(SHORT) == want and wx.wxpy_batch_shape_get(9) == (0, 4)
    doc["batch"].append({"bucket": 3, "tile": 0, "unroll_log2": 1, "built_in": 2})
    p.write_text(json.dumps(doc))
    with pytest.raises(wx.WxpyError):
        wx.wxpy_tune_cache_load(str(p), check_device=False)


def test_an_invalid_table_is_refused():
    with pytest.raises(wx.WxpyError) as e:
        vectors(wx.desc_table([8, 8], [1.0, 1.0], [B, B], [B, B], [B + 4096, B + 4096]))
    assert e.value.status == wx.WXPY_EOVERLAP
