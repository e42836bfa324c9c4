"""GPU parity of the batched entry points where their plan changes form: table
lengths around the plan's blocks and rounds, batches of one-tile segments
(warps walk runs of tiles) and of many-tile ones (warps stride), small batches
cut into short tiles, and segments whose pointers start at any element, alike
or each its own -- every element bit for bit."""
import numpy as np
import pytest
import torch

import paper_1309_1894_gb300 as wx
from paper_1309_1894_gb300 import binding, synth

pytestmark = pytest.mark.gpu


def run(entry, ns, seed, shifts):
    """Segments stored back to back in arenas that start `shifts` elements past
    an aligned address; the whole output arena, guards included."""
    total = int(sum(ns))
    starts = np.concatenate([[0], np.cumsum(ns)[:-1]]).astype(np.int64)
    alphas = synth.uniform_pm2(seed, synth.TAG_ALPHA, len(ns))
    xh, yh = (synth.uniform_pm1(seed, t, total) for t in (synth.TAG_X, synth.TAG_Y))
    x, y = (torch.empty(total + 4, dtype=torch.float64, device="cuda") for _ in range(2))
    w = torch.full((total + 8,), 7.25, dtype=torch.float64, device="cuda")
    x[shifts[0]:shifts[0] + total] = torch.from_numpy(xh).cuda()
    y[shifts[1]:shifts[1] + total] = torch.from_numpy(yh).cuda()
    table = wx.desc_table(ns, alphas, *(t.data_ptr() + 8 * (s + starts) for t, s in
                                        zip((x, y, w), shifts)))
    dev = wx.table_to_device(table)
    if entry == "noalloc":
        binding.wxpy_batch_noalloc(dev, len(ns))
    elif entry == "once":
        wx.wxpy_batch(table, dev)
    else:
        plan = wx.wxpy_batch_plan_create(table)
        plan.launch(dev)
        assert plan.status() == 0
    torch.cuda.synchronize()
    # two separately rounded operations, as the oracle's loop
    want = np.repeat(alphas, ns) * xh + yh
    got = w.cpu().numpy()
    assert np.array_equal(got[shifts[2]:shifts[2] + total].view(np.uint64), want.view(np.uint64))
    assert (got[:shifts[2]] == 7.25).all() and (got[shifts[2] + total:] == 7.25).all()


@pytest.mark.parametrize("entry", ["launch", "once", "noalloc"])
@pytest.mark.parametrize("count", [1, 2, 31, 33, 1023, 1025, 2048, 2049, 8193, 16385, 65536])
def test_table_lengths(entry, count):
    ns = synth.log_uniform_lengths(count, count, 1, 300)
    run(entry, ns, 40 + count, (0, 0, 0))


@pytest.mark.parametrize("entry", ["launch", "once", "noalloc"])
@pytest.mark.parametrize("shifts", [(0, 0, 0), (1, 1, 1), (0, 1, 2), (3, 0, 0)])
@pytest.mark.parametrize("lengths", [[70001], [1, 255, 256, 257, 5], [1 << 20, 1, 513],
                                     [31, 32, 33, 1000003, 8191, 8192, 8193], [5000] * 300])
def test_tiles_and_offsets(entry, lengths, shifts):
    run(entry, lengths, 90 + len(lengths), shifts)
