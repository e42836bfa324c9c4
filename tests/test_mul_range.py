"""The integer-pipeline product over its whole range of operands
(csrc/fp64_mul.cuh: mul_rn_range) against the host's IEEE multiplication, on
the CPU: exact wherever it is taken, and taken for every normal operand whose
product is in the normal range however it is rounded, at every coefficient
exponent."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
SIGS = [1.0, 1.0 + 2.0 ** -52, 1.5, 1.25, 2 ** 0.5, 2.0 - 2.0 ** -52, 1.9, 1.0 / 3 * 4]
DP = ctypes.POINTER(ctypes.c_double)


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("mulrange") / "libmul_range.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-ffp-contract=off", "-Wall",
                    "-Werror", os.path.join(HERE, "mul_range_check.cc"), "-o", so], check=True)
    L = ctypes.CDLL(so)
    L.mul_range_check.restype = ctypes.c_int64
    L.mul_range_check.argtypes = [ctypes.c_int64, ctypes.c_double, DP, ctypes.POINTER(ctypes.c_uint8)]
    L.mul_range_any.argtypes = [ctypes.c_int64, ctypes.c_double, DP]
    return L


def check(L, a, b):
    b = np.ascontiguousarray(b, np.float64)
    away = np.zeros(len(b), np.uint8)
    bad = L.mul_range_check(len(b), a, b.ctypes.data_as(DP),
                            away.ctypes.data_as(ctypes.POINTER(ctypes.c_uint8)))
    return bad, away.astype(bool)


def field(v):
    return ((np.ascontiguousarray(v, np.float64).view(np.uint64) >> np.uint64(52))
            & np.uint64(0x7FF)).astype(np.int64)


def test_taken_at_every_exponent(lib):
    eb = np.arange(-1022, 1024)
    for ea in range(-1022, 1024):
        a = float(np.ldexp(SIGS[ea % len(SIGS)], ea))
        b = np.ldexp(np.resize(SIGS, len(eb)), eb) * np.resize([1.0, -1.0, -1.0], len(eb))
        bad, away = check(lib, a, b)
        assert bad == 0
        # the product's exponent field, not counting a carry of the significands
        f = ea + eb + 1023
        assert np.array_equal(away, (f < 1) | (f > 2044)), ea


@pytest.mark.parametrize("a", [1.0, -0.7, 2.0 ** -300, -1.9e250, 2.0 ** 1023, 3e-308])
def test_random_and_specials(lib, a):
    rng = np.random.default_rng(61)
    b = np.ldexp(1 + rng.random(400_000), rng.integers(-1022, 1024, 400_000)) * rng.choice([-1, 1], 400_000)
    bad, away = check(lib, a, b)
    assert bad == 0 and not away.all()
    sv = np.array([0.0, -0.0, 5e-324, -2.2e-308, np.inf, -np.inf, np.nan])
    bad, away = check(lib, a, sv)
    assert bad == 0 and away.all()
    inside = b[~check(lib, a, b)[1]][:4]
    assert not lib.mul_range_any(4, a, inside.ctypes.data_as(DP))
    for v in sv:  # one of them takes the vector off the fast path, wherever it stands
        for k in range(4):
            u = inside.copy()
            u[k] = v
            assert lib.mul_range_any(4, a, u.ctypes.data_as(DP))


@pytest.mark.parametrize("a", [0.0, -0.0, 5e-324, np.inf, np.nan])
def test_coefficients_without_a_range(lib, a):
    bad, away = check(lib, a, np.ldexp(1.0, np.arange(-1022, 1024)))
    assert bad == 0 and away.all()
