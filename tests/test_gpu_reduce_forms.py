"""GPU parity of the fused reductions where the form of the call changes: the
cluster form with one and two columns per block, the block form on 32-byte
vectors, on vectors that start past the boundary and on single elements, and
the tree over the tile sums at every way it takes -- w and the result bit for
bit against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_1309_1894_gb300 as wx
from paper_1309_1894_gb300 import synth
from test_gpu_reduce import T, run, same_scalar, same_vec, want

pytestmark = pytest.mark.gpu

OFFS = [(0, 0, 0, 0), (8, 8, 8, 8), (16, 16, 16, 16), (24, 24, 24, 24), (0, 8, 16, 24)]


def inputs(n, seed):
    return (synth.uniform_pm1(seed, synth.TAG_X, n), synth.uniform_pm1(seed, synth.TAG_Y, n),
            synth.uniform_pm1(seed + 1, synth.TAG_X, n))


@pytest.mark.parametrize("offs", OFFS)
@pytest.mark.parametrize("n", [T - 127, 2 * T + 1, 33 * T - 3, 76 * T, 76 * T + 1, 256 * T - 130,
                               256 * T + 5, 1024 * T + 3])
def test_forms_at_their_edges(n, offs):
    xh, yh, zh = inputs(n, 700 + n % 97)
    for kind in ("norm2", "dot"):
        w, r = run(kind, 0.75, xh, yh, zh, offs)
        w_want, r_want = want(kind, 0.75, xh, yh, zh)
        assert same_vec(w, w_want) and same_scalar(r, r_want), (kind, n, offs)


@pytest.mark.parametrize("tiles", [1, 2, 3, 16, 32, 33, 64, 1024, 1025, 2048])
def test_signed_zero_sums(tiles):
    """Every term -0: the sum is -0 where the tree has no +0 padding, else +0."""
    n = tiles * T
    xh, zh = np.zeros(n), np.full(n, -1.0)
    _, r = run("dot", 1.0, xh, xh, zh, (0, 0, 0, 0))
    assert same_scalar(r, -0.0 if tiles & (tiles - 1) == 0 else 0.0)


def test_specials_and_coefficients_without_a_window():
    n = 77 * T + 9
    xh, yh, zh = inputs(n, 811)
    xh[::4097] = 0.0
    yh[::5003] = 0.0
    zh[1::3001] = 1e300
    xh[5::70001] = 1e-320
    for alpha in (0.0, -0.0, 5e-324, 1e308, 0.3):
        for kind in ("norm2", "dot"):
            for offs in ((0, 0, 0, 0), (8, 8, 8, 8), (8, 0, 8, 0)):
                with np.errstate(over="ignore", invalid="ignore"):
                    w_want, r_want = want(kind, alpha, xh, yh, zh)
                w, r = run(kind, alpha, xh, yh, zh, offs)
                assert same_vec(w, w_want) and same_scalar(r, r_want), (kind, alpha, offs)


@pytest.mark.parametrize("n", [5000, 20 * T, 300 * T])
def test_dependent_calls_back_to_back(n):
    """Each call reads what the one before wrote, with one workspace: a call
    whose launch overlaps the one before must still wait for it."""
    x, y, z = (torch.from_numpy(v).cuda() for v in inputs(n, 900))
    ws, res = wx.reduce_workspace(n), torch.empty(12, dtype=torch.float64, device="cuda")
    a, b = torch.empty_like(x), torch.empty_like(x)
    src, dst = x, a
    for k in range(12):
        wx.wxpy_dot(-0.5, src, y, z, w=dst, result=res[k:k + 1], workspace=ws)
        src, dst = dst, b if dst is a else a
    got = res.cpu().numpy()
    w, yh, zh = x.cpu().numpy(), y.cpu().numpy(), z.cpu().numpy()
    for k in range(12):
        w, r = oracle.wxpy_dot(-0.5, w, yh, zh)
        assert same_scalar(got[k], r), k
    assert same_vec(src.cpu().numpy(), w)


def test_more_tile_sums_than_the_threads_hold():
    n = 16384 * T + 1
    xh = synth.uniform_pm1(77, synth.TAG_X, 1 << 20)
    xh = np.resize(xh, n)
    x = torch.from_numpy(xh).cuda()
    w, r = wx.wxpy_norm2(0.25, x, x)
    torch.cuda.synchronize()
    w_want, r_want = oracle.wxpy_norm2(0.25, xh, xh)
    assert same_scalar(r.item(), r_want) and same_vec(w.cpu().numpy(), w_want)
