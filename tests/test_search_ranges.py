"""Searched choices by size range (no GPU): a split or a configuration found at
one size is used for calls of its range only, set and an older cache file apply
to every size, and the cache file keeps the ranges."""
import json

import pytest

import paper_1309_1894_gb300 as wx
from paper_1309_1894_gb300 import binding

SHORT, LONG = 10 ** 6, 1 << 24  # sibling kernels: below and from 2^23 elements
FEW, MANY = 1 << 21, (1 << 21) + 1  # reductions: the cluster form's tiles, and one more
split, config = binding.wxpy_debug_vecops_split, binding.wxpy_debug_reduce_config


@pytest.fixture(autouse=True)
def clear():
    wx.wxpy_tune_clear()
    yield
    wx.wxpy_tune_clear()


def load(tmp_path, vecops=(), reduce=()):
    p = tmp_path / "c.json"
    p.write_text(json.dumps({"format": "wxpy-tune-1", "device": "X", "vecops": list(vecops),
                             "reduce": list(reduce), "entries": []}))
    wx.wxpy_tune_cache_load(str(p), check_device=False)


def vec(cls, mul, **kw):
    return {"class": cls, "add_offload": 0, "mul_sixteenths": mul, **kw}


def red(kind, variant, levels=0, **kw):
    return {"kind": kind, "variant": variant, "mul_sixteenths": 16, "sum_levels": levels, **kw}


def test_a_long_calls_split_leaves_short_calls_alone(tmp_path):
    before = split(wx.VEC_AXPBY, SHORT)
    assert before == (0, 16)
    load(tmp_path, [vec(wx.VEC_AXPBY, 10, sizes=2)])
    assert split(wx.VEC_AXPBY, SHORT) == before and split(wx.VEC_AXPBY, (1 << 23) - 1) == before
    assert split(wx.VEC_AXPBY, 1 << 23) == split(wx.VEC_AXPBY, LONG) == (0, 10)
    assert wx.wxpy_vecops_tuned_get(wx.VEC_AXPBY) == (0, 10)
    load(tmp_path, [vec(wx.VEC_AXPBY, 14, sizes=1)])
    assert split(wx.VEC_AXPBY, SHORT) == (0, 14) and split(wx.VEC_AXPBY, LONG) == (0, 10)


def test_a_large_reductions_kernel_leaves_short_calls_the_cluster_form(tmp_path):
    before = [config(k, FEW) for k in (0, 1)]
    assert before == [(0, 16, 0), (0, 16, 0)]
    load(tmp_path, (), [red(0, 5, 2, sizes=2), red(1, 3, sizes=2)])
    assert [config(k, FEW) for k in (0, 1)] == before
    assert config(0, MANY) == (5, 16, 2) and config(1, MANY) == (3, 16, 0)


def test_set_and_entries_without_a_range_apply_to_every_size(tmp_path):
    wx.wxpy_vecops_tuned_set(3, 1, 6)
    wx.wxpy_reduce_tuned_set(0, 2, 8, 0)
    assert split(3, SHORT) == split(3, LONG) == (1, 6)
    assert config(0, FEW) == config(0, MANY) == (2, 8, 0)
    wx.wxpy_tune_clear()
    load(tmp_path, [vec(3, 4)], [red(1, 1)])
    assert split(3, SHORT) == split(3, LONG) == (0, 4)
    assert config(1, FEW) == config(1, MANY) == (1, 16, 0)
    wx.wxpy_vecops_tuned_set(3, -1, -1)
    assert split(3, SHORT) == split(3, LONG) == (0, 16)


def test_a_knob_wins_over_both_ranges(tmp_path):
    load(tmp_path, [vec(0, 6, sizes=1), vec(0, 8, sizes=2)], [red(0, 4, sizes=1), red(0, 5, sizes=2)])
    wx.wxpy_vecops_pipes(-1, 3)
    wx.wxpy_reduce_variant(1)
    try:
        assert split(0, SHORT) == split(0, LONG) == (0, 3)
        assert config(0, FEW)[0] == config(0, MANY)[0] == 1
    finally:
        wx.wxpy_vecops_pipes(-1, -1)
        wx.wxpy_reduce_variant(-1)
    assert split(0, SHORT) == (0, 6) and split(0, LONG) == (0, 8)


@pytest.mark.parametrize("sizes", [0, 3, -1])
def test_a_malformed_range_stores_nothing(tmp_path, sizes):
    for kw in ({"vecops": [vec(2, 6), vec(3, 6, sizes=sizes)]},
               {"reduce": [red(0, 2), red(1, 2, sizes=sizes)]}):
        with pytest.raises(wx.WxpyError):
            load(tmp_path, **kw)
    assert wx.wxpy_vecops_tuned_get(2) == (-1, -1) and wx.wxpy_reduce_tuned_get(0) == (-1, -1, -1)
