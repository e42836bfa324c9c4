"""The windowed integer-pipeline sum (csrc/fp64_emu.cuh: add_rn_quick) against
the host's IEEE addition, on the CPU: every exponent gap, both signs, ties,
carries, cancellations and special operands -- exact wherever it is taken, and
taken on the documented domain."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("addquick") / "libadd_quick.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-ffp-contract=off", "-Wall",
                    "-Werror", os.path.join(HERE, "add_quick_check.cc"), "-o", so], check=True)
    L = ctypes.CDLL(so)
    dp = ctypes.POINTER(ctypes.c_double)
    L.add_quick_check.restype = ctypes.c_int64
    L.add_quick_check.argtypes = [ctypes.c_int64, dp, dp, ctypes.POINTER(ctypes.c_uint8)]

    def run(a, b):
        a, b = (np.ascontiguousarray(v, np.float64) for v in (a, b))
        away = np.zeros(len(a), np.uint8)
        bad = L.add_quick_check(len(a), a.ctypes.data_as(dp), b.ctypes.data_as(dp),
                                away.ctypes.data_as(ctypes.POINTER(ctypes.c_uint8)))
        return bad, away.astype(bool)
    return run


def field(v):
    return ((np.abs(v).view(np.uint64) >> np.uint64(52)) & np.uint64(0x7FF)).astype(np.int64)


@pytest.mark.parametrize("signs", [1.0, -1.0])
def test_every_gap(check, signs):
    rng = np.random.default_rng(51)
    m = 20000
    for gap in [*range(0, 70), 95, 96, 97, 127, 128, 400, 900]:
        e = rng.integers(-400, 400, m) if gap < 500 else rng.integers(0, 900, m)
        a = np.ldexp(1 + rng.random(m), e)
        b = signs * np.ldexp(1 + rng.random(m), e - gap)
        short = signs * np.ldexp(1 + rng.integers(0, 8, m) / 8.0, e - gap)  # ties at gaps near 53
        for x, y in ((a, b), (b, a), (-a, -b), (a, short), (short, a)):
            bad, away = check(x, y)
            assert bad == 0, gap
            if signs > 0 or gap > 1:
                assert not away.any()
            else:  # cancellation leaves the fast path only when it is deep
                assert away.mean() < 2.0 ** -12 or gap == 0 and away.mean() < 0.2


def test_ties_carries_and_cancellations(check):
    rng = np.random.default_rng(52)
    m = 100_000
    k = rng.integers(1 << 52, 1 << 53, m)
    a = k.astype(np.float64) * 2.0 ** -52
    for gap in range(1, 31):
        # b = odd multiple of half an ulp of a, and just beside it
        odd = (2 * rng.integers(1 << (51 - gap), 1 << (52 - gap), m) + 1).astype(np.float64)
        for off in (0.0, 2.0 ** -60, -(2.0 ** -60)):
            b = odd * 2.0 ** -53 + off
            for x, y in ((a, b), (-a, b), (a, -b)):
                assert check(x, y)[0] == 0
    ones = np.full(m, 2.0 - 2.0 ** -52)
    assert check(ones, rng.integers(1, 4096, m) * 2.0 ** -53)[0] == 0
    near = a * (1 - rng.integers(0, 1 << 30, m) * 2.0 ** -52)
    bad, _ = check(a, -near)
    assert bad == 0
    bad, away = check(a, -a)
    assert bad == 0 and away.all()  # exact zero goes to the hardware
    bad, away = check(a, a)
    assert bad == 0 and not away.any()


def test_window_and_specials(check):
    sv = [0.0, -0.0, 5e-324, 2.2e-308, np.inf, -np.inf, np.nan, 1.0, -1.0, 1.5]
    sv += [s * np.ldexp(f, e) for e in (-512, -511, -510, 510, 511, 512, 513, 1023, -1022,
                                        -960, -959, -958, 991, 992, 993)
           for f in (1.0, 1.75) for s in (1, -1)]
    a, b = (v.astype(np.float64) for v in (np.repeat(sv, len(sv)), np.tile(sv, len(sv))))
    with np.errstate(all="ignore"):
        bad, away = check(a, b)
    hi = np.maximum(field(a), field(b))
    assert bad == 0
    assert away[(hi < 64) | (hi > 2015)].all()
    gap = np.abs(field(a) - field(b))
    same = np.signbit(a) == np.signbit(b)
    assert not away[(hi >= 64) & (hi <= 2015) & (same | (gap > 1))].any()


@pytest.mark.parametrize("gap", [31, 32, 33, 34, 52, 53, 54, 55, 62, 63, 64, 65, 200])
def test_one_lost_bit_decides(check, gap):
    """A smaller operand of few bits below the last one of the larger: ties, and
    ties missed by its lowest bit alone, added and subtracted, the larger one a
    power of two (whose difference has one bit more) or just beside it."""
    a, b = [], []
    for hi in (1.0, 1.0 + 2.0 ** -52, 1.0 + 2.0 ** -51, 1.5, 2.0 - 2.0 ** -52):
        for lo in (1.0, 1.0 + 2.0 ** -52, 1.5, 1.0 + 2.0 ** -31, 1.0 + 2.0 ** -20, 2.0 - 2.0 ** -52):
            for e in (0, 300, -300):
                a.append(np.ldexp(hi, e))
                b.append(np.ldexp(lo, e - gap))
    a, b = np.array(a), np.array(b)
    for x, y in ((a, b), (a, -b), (-a, b), (-b, a), (b, -a)):
        bad, away = check(x, y)
        assert bad == 0 and not away.any()


def test_zero_and_subnormal_addends(check):
    a = np.ldexp(1.0 + np.arange(64) * 2.0 ** -52, np.arange(64) * 30 - 959)
    for z in (0.0, -0.0, 5e-324, -2.2e-308):
        b = np.full(64, z)
        for x, y in ((a, b), (b, a), (-a, b)):
            bad, away = check(x, y)
            assert bad == 0 and not away.any()
