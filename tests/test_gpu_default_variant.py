"""wxpy() with the untuned variant at the sizes where that variant changes.

The variant of a call that no search has covered depends on the size and on the
pointers' class; every one of them has to give the bits of the plain reference
kernel (paper 1309.1894, Fig. 1: w = alpha*x + y, each operation rounded once),
at the last size of one range and the first of the next.
"""

import pytest
import torch

import paper_1309_1894_gb300 as wx
from gpu_util import Guarded, dev_bits_equal
from paper_1309_1894_gb300 import synth

pytestmark = pytest.mark.gpu

EDGES = [4096, 4097, 1 << 15, (1 << 15) + 1, 1 << 17, (1 << 17) + 1, 3 << 18, (3 << 18) + 1,
         1 << 20, (1 << 20) + 1, 152 * 8 * 1024, 152 * 8 * 1024 + 1, (1 << 23) - 1, 1 << 23,
         (1 << 25) - 1, 1 << 25]
# offsets of x, y, w in bytes: one class of pointers each
CLASSES = [("distinct", (0, 0, 0)), ("distinct", (8, 8, 8)), ("distinct", (16, 0, 16)),
           ("distinct", (8, 24, 0)), ("w=x", (8, 8, 8)), ("x=y", (0, 0, 0)),
           ("x=y", (24, 24, 8)), ("x=y", (8, 8, 16))]


@pytest.mark.parametrize("alias,offs", CLASSES, ids=lambda v: str(v))
@pytest.mark.parametrize("n", EDGES)
def test_untuned_variant_at_the_edges_of_its_ranges(n, alias, offs):
    wx.wxpy_tune_clear()
    gx, gy, gw = (Guarded(n, o) for o in offs)
    wx.wxpy_fill_uniform(gx.t, n, synth.TAG_X)
    wx.wxpy_fill_uniform(gy.t, n, synth.TAG_Y)
    x = gx.t
    y = x if alias == "x=y" else gy.t
    w = x if alias == "w=x" else gw.t
    want = torch.empty(n, dtype=torch.float64, device="cuda")
    wx.wxpy_reference(-0.7310585786300049, x, y, want)
    wx.wxpy(-0.7310585786300049, x, y, w)
    torch.cuda.synchronize()
    assert wx.wxpy_lookup(x, y, w)[1] == 0  # untuned
    assert dev_bits_equal(w, want)
    for g in (gx, gy, gw):
        g.check()
