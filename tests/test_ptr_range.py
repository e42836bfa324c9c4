"""Which source ranges the server hands to a kernel (csrc/ptr_range.h), on the
CPU against a made-up address space: a copy call refuses a range that is not
inside one allocation, a kernel would fault on it, so such a range must go to
the copy call.  No launch is made with one."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
A, B, H, M, R = 0x7F0000000000, 0x7F0000400000, 0x10000000, 0x7F1000000000, 0x7F2000000000
# mapped from, mapped bytes, reported start and size, plain device memory, device
ROWS = np.array([
    [A, 1 << 20, A, 1 << 20, 1, 0],        # an allocation
    [A + (1 << 20), 4096, A + (1 << 20), 4096, 1, 0],  # its neighbour, with no gap between
    [B, 1 << 20, B, 1 << 20, 1, 1],        # another device's
    [H, 1 << 20, H, 1 << 20, 0, 0],        # host memory
    [M, 1 << 20, M, 1 << 20, 0, 0],        # managed memory
    [R, 1 << 16, R, 1 << 24, 1, 0],        # a reservation, mapped at its start only
], np.uint64)


@pytest.fixture(scope="module")
def inside(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("ptrrange") / "libptr_range.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-Wall", "-Werror",
                    os.path.join(HERE, "ptr_range_check.cc"), "-o", so], check=True)
    f = ctypes.CDLL(so).range_check
    f.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_uint64, ctypes.c_uint64, ctypes.c_int]
    return lambda p, n_bytes, device=0: bool(f(ROWS.ctypes.data, len(ROWS), p, n_bytes, device))


@pytest.mark.parametrize("p,n_bytes", [(A, 8), (A, 1 << 20), (A + 8, (1 << 20) - 8),
                                       (A + (1 << 20) - 8, 8), (R, 1 << 16)])
def test_taken(inside, p, n_bytes):
    assert inside(p, n_bytes)


@pytest.mark.parametrize("p,n_bytes", [
    (A, (1 << 20) + 8),              # one element past the end, into the neighbour
    (A + 8, 1 << 20),
    (A, 1 << 40),                    # a wrong length
    (A, 2 ** 64 - 8),                # .. that wraps around
    (A - 8, 16),                     # before the start
    (A + (1 << 22), 8),              # nothing there (a freed buffer)
    (B, 8), (H, 8), (M, 8),          # not plain memory of this device
    (R, (1 << 16) + 8),              # reserved, not mapped
    (A, 0),
])
def test_left_to_the_copy_call(inside, p, n_bytes):
    assert not inside(p, n_bytes)
