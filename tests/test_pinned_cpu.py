"""The bounded free list of page-locked buffers (csrc/zmc_pinned.h)."""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture
def pool(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no g++")
    so = str(tmp_path / "pool.so")
    subprocess.run([gxx, "-O1", "-std=c++17", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_1910_01965_gb300", "csrc"), "-o", so,
                    os.path.join(ROOT, "tests", "pinned_wrap.cpp")], check=True)
    L = ctypes.CDLL(so)
    L.pool_new.restype = ctypes.c_void_p
    L.pool_new.argtypes = [ctypes.c_size_t]
    L.pool_take.argtypes = [ctypes.c_void_p, ctypes.c_size_t, ctypes.POINTER(ctypes.c_void_p),
                            ctypes.POINTER(ctypes.c_size_t)]
    L.pool_give.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_size_t]

    def take(h, n):
        p, got = ctypes.c_void_p(), ctypes.c_size_t()
        assert L.pool_take(h, n, ctypes.byref(p), ctypes.byref(got)) == 0
        return p.value, got.value

    L.take = take
    return L


def test_small_takes_leave_large_buffers(pool):
    h = pool.pool_new(4)
    bufs = [pool.take(h, n) for n in (1 << 26, 1 << 18, 1 << 20)]
    for p, n in bufs:
        pool.pool_give(h, p, n)
    assert pool.take(h, 1 << 18) == bufs[1]          # the smallest that fits
    assert pool.take(h, 1 << 18) == bufs[2]
    assert pool.take(h, (1 << 20) + 1) == bufs[0]
    assert pool.pool_made() == 3


def test_bounded_and_reused(pool):
    h = pool.pool_new(32)
    for turn in range(3):
        held = [pool.take(h, 1 << 18) for _ in range(40)]
        assert len({p for p, _ in held}) == 40
        for p, n in held:
            pool.pool_give(h, p, n)
        assert pool.pool_live() == 32                # the rest was given back
    assert pool.pool_made() == 40 + 8 + 8


def test_errors_come_back(pool):
    h = pool.pool_new(4)
    pool.pool_fail(2)
    p, got = ctypes.c_void_p(), ctypes.c_size_t(7)
    assert pool.pool_take(h, 64, ctypes.byref(p), ctypes.byref(got)) == 2
    assert p.value is None and got.value == 0
