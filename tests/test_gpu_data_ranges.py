"""GPU parity on data that leaves the integer products' fast path: zeros,
infinities, NaNs and subnormals among ordinary values, magnitudes over the whole
exponent range, and coefficients at its ends -- every element bit for bit (a NaN
for a NaN)."""
import numpy as np
import pytest
import torch

import oracle
import paper_1309_1894_gb300 as wx
from paper_1309_1894_gb300 import binding, synth

pytestmark = pytest.mark.gpu

KINDS = ["zeros", "sevenths", "infinite", "mixed", "huge", "tiny", "spread"]


def data(kind, n, seed):
    """Values of one kind; the rest U(-1, 1)."""
    v = synth.uniform_pm1(seed, synth.TAG_X, n)
    rng = np.random.default_rng(seed)
    if kind == "zeros":
        v[:] = 0.0
        v[1::2] = -0.0
    elif kind == "sevenths":
        v[::7] = 0.0
    elif kind == "infinite":
        v[:] = np.inf
    elif kind == "mixed":
        at = rng.permutation(n)
        for k, s in enumerate((0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, -1e-310, 1e300, -1e-300)):
            v[at[k * (n // 97):(k + 1) * (n // 97)]] = s
    elif kind == "huge":
        v *= 1e200
    elif kind == "tiny":
        v *= 1e-200
    elif kind == "spread":
        v = np.ldexp(v, rng.integers(-1070, 1024, n))
    return v


def same(got, want):
    got, want = (np.ascontiguousarray(a, np.float64) for a in (got, want))
    nan = np.isnan(want)
    return np.array_equal(np.isnan(got), nan) and \
        np.array_equal(got.view(np.uint64)[~nan], want.view(np.uint64)[~nan])


def at(host, shift):
    t = torch.empty(len(host) + 8, dtype=torch.float64, device="cuda")[shift:shift + len(host)]
    return t.copy_(torch.from_numpy(host))


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("shifts", [(0, 0, 0), (2, 0, 2), (0, 1, 3), (1, 1, 1)])
@pytest.mark.parametrize("n", [1027, 100003, (1 << 20) + 1])
def test_single_calls(n, shifts, kind):
    xh, yh = data(kind, n, 21 + n % 13), synth.uniform_pm1(5, synth.TAG_Y, n)
    x, y = at(xh, shifts[0]), at(yh, shifts[1])
    for alpha in (0.7, -2.0 ** 600, 3e-308, 1e308, 0.0):
        with np.errstate(all="ignore"):
            want, want_xx = oracle.wxpy(alpha, xh, yh), oracle.wxpy(alpha, xh, xh)
        w = at(np.zeros(n), shifts[2])
        wx.wxpy(alpha, x, y, w)
        assert same(w.cpu().numpy(), want), alpha
        wx.wxpy(alpha, x, x, w)
        assert same(w.cpu().numpy(), want_xx), alpha


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("entry", ["launch", "once", "noalloc"])
@pytest.mark.parametrize("shifts", [(0, 0, 0), (3, 0, 1)])
@pytest.mark.parametrize("lengths", [[5, 1, 70001, 4099], [300] * 500, [40000] * 260])
def test_batches(entry, kind, shifts, lengths):
    total = sum(lengths)
    starts = np.concatenate([[0], np.cumsum(lengths)[:-1]]).astype(np.int64)
    xh, yh = data(kind, total, 31), synth.uniform_pm1(6, synth.TAG_Y, total)
    alphas = np.resize([0.7, -2.0 ** 600, 3e-308, 1e308, 0.0, -0.3], len(lengths))
    x, y, w = at(xh, shifts[0]), at(yh, shifts[1]), at(np.full(total, 7.25), shifts[2])
    table = wx.desc_table(lengths, alphas, *(t.data_ptr() + 8 * starts for t in (x, y, w)))
    dev = wx.table_to_device(table)
    if entry == "noalloc":
        binding.wxpy_batch_noalloc(dev, len(lengths))
    elif entry == "once":
        wx.wxpy_batch(table, dev)
    else:
        wx.wxpy_batch_plan_create(table).launch(dev)
    torch.cuda.synchronize()
    with np.errstate(all="ignore"):
        want = np.repeat(alphas, lengths) * xh + yh  # two roundings, as the oracle's loop
    assert same(w.cpu().numpy(), want)


# Lengths: less than a tile per SM; several tiles per warp, so that warps switch
# to FP64 products or sums and back.
@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("n,shifts", [(4099, (0, 0, 0)), (100003, (0, 1, 2)), (6_000_001, (1, 1, 1)),
                                      (6_000_001, (0, 1, 0))])
def test_streaming_siblings(n, shifts, kind):
    xh, yh, zh = (data(k, n, 41 + j) for j, k in enumerate((kind, "uniform", "uniform")))
    x, y, z = (at(v, s) for v, s in zip((xh, yh, zh), shifts))
    for c in ((0.7, -0.2, 0.3), (2.0 ** 600, 1e-300, -1.0), (0.5, 0.0, 1e308)):
        with np.errstate(all="ignore"):
            want2, want3 = oracle.axpby(c[0], c[1], xh, yh), oracle.axpbypcz(*c, xh, yh, zh)
        y2, z3 = at(yh, shifts[1]), at(zh, shifts[2])
        wx.wxpy_axpby(c[0], c[1], x, y2)
        wx.wxpy_axpbypcz(*c, x, y, z3)
        assert same(y2.cpu().numpy(), want2) and same(z3.cpu().numpy(), want3), c
    wx.wxpy_vecops_status()  # no wait ran out


@pytest.mark.parametrize("m", [2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("kind,scale", [("uniform", 1e-12), ("uniform", 2.0 ** -31), ("uniform", 1e12),
                                        ("y zero", 1.0), ("y infinite", 1.0), ("cancelling", 1.0),
                                        ("mixed", 1.0), ("sevenths", 1e-12), ("spread", 1.0),
                                        ("ties", 1.0)])
@pytest.mark.parametrize("n,shifts", [(4099, (0, 0)), (2_000_003, (0, 0)), (2_000_003, (1, 0))])
def test_maxpy_sums(n, shifts, m, kind, scale):
    """Terms far below and above the vector they are added to, a zero vector, and
    sums that cancel: the integer sums leave their path in some elements or all."""
    special = kind if kind in KINDS else "uniform"
    xs = [data(special if j == 1 else "uniform", n, 51 + j) * scale for j in range(m)]
    yh = data("uniform", n, 50)
    al = [0.75, -1.5, 1.25, -0.625, 1.875, -0.3125, 0.5625, -1.0625][:m]
    if kind == "y zero":
        yh[:] = 0.0
        yh[::3] = -0.0
    elif kind == "y infinite":
        yh[1::5] = np.inf
    elif kind == "ties":
        # half an ulp of the sum so far, exactly or missed by a bit far below, at gaps
        # of 52 to 54 and beyond
        rng = np.random.default_rng(n + m)
        yh = (1.0 + rng.integers(0, 1 << 52, n) * 2.0 ** -52) * np.where(rng.random(n) < 0.1, 0, 1) + 1.0
        al = [1.0, -1.0, 0.5, 2.0, -0.5, 1.0, -2.0, 0.25][:m]
        for j in range(m):
            half = 2.0 ** -52 * rng.choice([0.5, 1.0, 1.5, 2.0, 3.0, 2.0 ** -8], n)
            xs[j] = half * (1 + rng.choice([0.0, 2.0 ** -52, 2.0 ** -20, -2.0 ** -53], n))
            xs[j] *= rng.choice([-1.0, 1.0], n)
    elif kind == "cancelling":
        for j in range(1, m):
            xs[j][::2] = xs[j - 1][::2] * (-al[j - 1] / al[j]) * (1 + 2.0 ** -40)
    with np.errstate(all="ignore"):
        want = oracle.maxpy(al, xs, yh)
    y = at(yh, shifts[0])
    wx.wxpy_maxpy(al, [at(v, shifts[1]) for v in xs], y)
    assert same(y.cpu().numpy(), want)
    wx.wxpy_vecops_status()  # no wait ran out


# Tiles of 8192 elements: the cluster form; the block form with one tile and with
# a few per block, whose later tiles take other products where the earlier ones
# left the integer pipelines; every way the offsets deal the elements.
@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("tiles", [2, 130, 300, 1000, 2500])
@pytest.mark.parametrize("shifts", [(0, 0, 0, 0), (1, 1, 1, 1), (0, 1, 2, 3)])
def test_reductions(tiles, shifts, kind):
    n = tiles * 8192 - 100
    xh, yh, zh = (data(k, n, 61 + j) for j, k in enumerate((kind, "uniform", "uniform")))
    x, y, z = (at(v, s) for v, s in zip((xh, yh, zh), shifts))
    w = at(np.zeros(n), shifts[3])
    for alpha in (0.7, 0.0) if tiles > 1000 else (0.7, -2.0 ** 600, 3e-308, 0.0):
        with np.errstate(all="ignore"):
            (w2, n2), (w3, d3) = oracle.wxpy_norm2(alpha, xh, yh), oracle.wxpy_dot(alpha, xh, yh, zh)
        _, r = wx.wxpy_norm2(alpha, x, y, w=w)
        assert same(w.cpu().numpy(), w2) and same(r.cpu().numpy(), np.array([n2])), alpha
        _, r = wx.wxpy_dot(alpha, x, y, z, w=w)
        assert same(w.cpu().numpy(), w3) and same(r.cpu().numpy(), np.array([d3])), alpha


@pytest.mark.parametrize("shifts", [(0, 0, 0, 0), (1, 1, 1, 1), (0, 1, 2, 3)])
def test_reductions_change_products_and_back(shifts):
    """A stretch of zeros, one of infinities, ordinary data before, between and
    after: every block meets each, and the terms' products leave in one alone."""
    n = 5000 * 8192 + 7
    xh, yh, zh = (data("uniform", n, 71 + j) for j in range(3))
    xh[n // 5:2 * n // 5] = 0.0
    xh[n // 2:n // 2 + 100] = np.inf
    zh[3 * n // 5:4 * n // 5:2] = 0.0
    yh[n // 5:n // 4] = 0.0
    x, y, z = (at(v, s) for v, s in zip((xh, yh, zh), shifts))
    w = at(np.zeros(n), shifts[3])
    with np.errstate(all="ignore"):
        (w2, n2), (w3, d3) = oracle.wxpy_norm2(0.7, xh, yh), oracle.wxpy_dot(0.7, xh, yh, zh)
    for mul in (-1, 16, 8):
        wx.wxpy_reduce_pipes(mul)
        try:
            _, r = wx.wxpy_norm2(0.7, x, y, w=w)
            assert same(w.cpu().numpy(), w2) and same(r.cpu().numpy(), np.array([n2])), mul
            _, r = wx.wxpy_dot(0.7, x, y, z, w=w)
            assert same(w.cpu().numpy(), w3) and same(r.cpu().numpy(), np.array([d3])), mul
        finally:
            wx.wxpy_reduce_pipes(-1)
