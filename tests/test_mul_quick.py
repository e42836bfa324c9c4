"""The windowed integer-pipeline products (csrc/fp64_mul.cuh: mul_rn_quick,
mul_rn_quick2) against the host's IEEE multiplication, on the CPU: exact
wherever they are taken, taken exactly on the documented exponent windows, at
every coefficient exponent; ties, carries and special operands included."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("mulquick") / "libmul_quick.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-ffp-contract=off", "-Wall",
                    "-Werror", os.path.join(HERE, "mul_quick_check.cc"), "-o", so], check=True)
    L = ctypes.CDLL(so)
    dp = ctypes.POINTER(ctypes.c_double)
    L.mul_quick_check.restype = ctypes.c_int64
    L.mul_quick_check.argtypes = [ctypes.c_int64, dp, dp, ctypes.c_int,
                                  ctypes.POINTER(ctypes.c_uint8)]
    L.mul_window.argtypes = [ctypes.c_double]
    return L


def check(L, a, b, two):
    a, b = (np.ascontiguousarray(v, np.float64) for v in (a, b))
    away = np.zeros(len(a), np.uint8)
    dp = ctypes.POINTER(ctypes.c_double)
    with np.errstate(all="ignore"):
        bad = L.mul_quick_check(len(a), a.ctypes.data_as(dp), b.ctypes.data_as(dp), two,
                                away.ctypes.data_as(ctypes.POINTER(ctypes.c_uint8)))
    return bad, away.astype(bool)


def field(v):
    return ((np.ascontiguousarray(v, np.float64).view(np.uint64) >> np.uint64(52))
            & np.uint64(0x7FF)).astype(np.int64)


SIGS = [1.0, 1.0 + 2.0 ** -52, 1.5, 1.25, 2 ** 0.5, 2.0 - 2.0 ** -52, 1.9, 1.0 / 3 * 4]


@pytest.mark.parametrize("two", [0, 1])
def test_random_ties_and_carries(lib, two):
    rng = np.random.default_rng(31)
    m = 200_000
    a = np.ldexp(1 + rng.random(m), rng.integers(-300, 300, m)) * rng.choice([-1.0, 1.0], m)
    b = np.ldexp(1 + rng.random(m), rng.integers(-200, 200, m)) * rng.choice([-1.0, 1.0], m)
    short = np.ldexp(1 + rng.integers(0, 1 << 6, m) * 2.0 ** -6, rng.integers(-9, 9, m))
    for x, y in ((a, b), (b, short), (short, b), (short, short),
                 (np.full(m, 2.0 - 2.0 ** -52), 1 + rng.integers(0, 4096, m) * 2.0 ** -52)):
        bad, away = check(lib, x, y, two)
        assert bad == 0 and not away.any()


def test_coefficient_window_at_every_exponent(lib):
    """Every product inside the window is exact and in the normal range; the
    window is 1024 fields wide; operands outside it leave the fast path."""
    eb = np.arange(-1074, 1025)
    for ea in range(-1022, 1024):
        a = np.ldexp(SIGS[ea % len(SIGS)], ea)
        first = lib.mul_window(a)
        assert (first == 0) == (abs(a) >= 2.0 ** 1021), ea
        if first == 0:
            continue
        with np.errstate(over="ignore"):
            b = np.ldexp(SIGS[(ea * 5 + 3) % len(SIGS)], eb)
        bad, away = check(lib, np.full(len(b), -a), b, 0)
        f = field(b)
        assert bad == 0
        assert np.array_equal(away, (f < first) | (f > first + 1023))


def test_two_operand_window_and_specials(lib):
    sv = [0.0, -0.0, 5e-324, 2.2e-308, np.inf, -np.inf, np.nan, 1.0, -3.0]
    sv += [np.ldexp(s, e) for s in SIGS for e in (-512, -511, -510, 511, 512, 513, 1023, -1022)]
    a, b = np.repeat(sv, len(sv)), np.tile(sv, len(sv))
    bad, away = check(lib, a, b, 1)
    inside = [(field(v) >= 512) & (field(v) <= 1534) for v in (a, b)]
    assert bad == 0 and np.array_equal(away, ~(inside[0] & inside[1]))
    for v in (0.0, -0.0, 5e-324, np.inf, np.nan):
        assert lib.mul_window(v) == 0
