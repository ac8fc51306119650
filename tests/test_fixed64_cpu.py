"""The 64-bit fixed-point arithmetic of the FP64 integrands (csrc/zmc_fixed64.cuh),
compiled with the host compiler and compared with high-precision arithmetic."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

mpmath = pytest.importorskip("mpmath")
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
i64, u64, u32, f64 = ctypes.c_int64, ctypes.c_uint64, ctypes.c_uint32, ctypes.c_double


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no g++")
    so = str(tmp_path_factory.mktemp("fx") / "fx.so")
    subprocess.run([gxx, "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_1910_01965_gb300", "csrc"), "-o", so,
                    os.path.join(ROOT, "tests", "fixed64_wrap.cpp")], check=True)
    L = ctypes.CDLL(so)
    L.fx_cos_table.restype = L.fx_exp_table.restype = ctypes.POINTER(i64)
    L.fx_phase.restype, L.fx_phase.argtypes = u64, [u64, u32, ctypes.c_void_p]
    L.fx_scale.restype, L.fx_scale.argtypes = i64, [f64, u64]
    L.fx_sum.restype = f64
    mpmath.mp.prec = 400
    return L


def _call(fn, dtype, n, *arrays):
    out = np.empty(n, dtype)
    fn(*[a.ctypes.data_as(ctypes.c_void_p) for a in arrays],
       out.ctypes.data_as(ctypes.c_void_p), ctypes.c_int(len(arrays[0])))
    return out


def test_tables(lib):
    c, e = lib.fx_cos_table(), lib.fx_exp_table()
    for i in range(2560):
        x = mpmath.cos(2 * mpmath.pi * i / 2048) * 2 ** 62
        assert abs(c[i] - 2 ** 31 - x) <= 0.5
    for i in range(2048):
        assert abs(e[i] - 2 ** 31 - mpmath.mpf(2) ** (62 - mpmath.mpf(i) / 2048)) <= 0.5


def _angles():
    r = np.random.default_rng(1)
    th = r.integers(0, 2 ** 64, 3000, dtype=np.uint64)
    step = np.arange(0, 2048, 7, dtype=np.uint64) << np.uint64(53)
    edge = [step, step - np.uint64(1), step + np.uint64(1 << 52),
            step + np.uint64((1 << 52) - 1), step + np.uint64((1 << 53) - 1)]
    return np.concatenate([th] + edge)


def test_cos(lib):
    """Within 2^-56 (an FP64 rounding near 1 is 2^-54), and unbiased: the mean
    error within five standard errors of zero."""
    th = _angles()
    got = _call(lib.fx_cos_n, np.int64, len(th), th)
    err = np.array([float(int(g) * mpmath.mpf(2) ** -62 - mpmath.cos(
        2 * mpmath.pi * (mpmath.mpf(int(t)) * mpmath.mpf(2) ** -64 - mpmath.mpf(2) ** -12)))
        for t, g in zip(th, got)])
    assert np.max(np.abs(err)) < 2.0 ** -56
    rnd = err[:3000]
    assert abs(rnd.mean()) < 5 * rnd.std() / np.sqrt(len(rnd))


def test_exp2neg(lib):
    """Relative error below 2^-52.5: half a unit in the last place from the final
    rounding (2^-53) and 2^-54.2 from the evaluation."""
    r = np.random.default_rng(2)
    half = 1 << 42
    q = [int(v) for v in r.integers(half, 1000 << 54, 3000, dtype=np.uint64)]
    q += [int(v) for v in r.integers(half, 8 << 54, 3000, dtype=np.uint64)]
    for i in range(0, 2049, 9):  # both ends of a table step, and whole powers of two
        q += [(i << 43) + o for o in (half, half - 1 + (1 << 43), half + (1 << 42))]
    q = np.array([v for v in q if v >= half], np.uint64)
    got = _call(lib.fx_exp_n, np.float64, len(q), q)
    err = []
    for a, g in zip(q, got):
        x = mpmath.mpf(2) ** (-(mpmath.mpf(int(a)) * mpmath.mpf(2) ** -54 - mpmath.mpf(2) ** -12))
        err.append(float((mpmath.mpf(float(g)) - x) / x))
    assert np.max(np.abs(err)) < 2.0 ** -52.5
    assert got[np.flatnonzero(q == half)[0]] == 1.0


def test_mul62(lib):
    r = np.random.default_rng(3)
    a = r.integers(-2 ** 62, 2 ** 62, 4000)
    b = r.integers(-2 ** 62, 2 ** 62, 4000)
    a[:4] = [2 ** 62, 2 ** 62, -2 ** 62, 0]
    b[:4] = [2 ** 62, -2 ** 62, -2 ** 62, 5]
    got = _call(lib.fx_mul62_n, np.int64, len(a), a, b)
    err = [abs((int(g) << 62) - int(x) * int(y)) / 2 ** 62 for g, x, y in zip(got, a, b)]
    assert max(err) <= 6.0  # of 2^-62


def test_turns_and_phase(lib):
    r = np.random.default_rng(4)
    c = r.uniform(-1, 1, 400) * 2.0 ** r.integers(-200, 30, 400)
    c[:6] = [0.0, -0.0, 5e-324, 1e-300, 2.0 ** 29, -(2.0 ** 30 - 2.0 ** -23)]
    k = np.zeros(400, np.int32)
    k[50:] = r.integers(-60, 1, 350)
    t = _call(lib.fx_turns_n, np.uint32, 1200, c, k).reshape(-1, 3)
    one = 2 ** 96
    for ci, ki, w in zip(c, k, t):
        want = mpmath.mpf(float(ci)) * mpmath.mpf(2) ** int(ki) / (2 * mpmath.pi) * one
        got = int(w[0]) + (int(w[1]) << 32) + (int(w[2]) << 64)
        d = (got - want) % one
        assert min(d, one - d) <= 2
        v = int(r.integers(0, 2 ** 23))
        th = lib.fx_phase(12345, v, np.ascontiguousarray(w).ctypes.data)
        d = (th - 12345 - mpmath.mpf(got) * v / 2 ** 32) % 2 ** 64
        assert min(d, 2 ** 64 - d) <= 2


def test_scale59(lib):
    K = 0x5a9825b501cd145c
    assert abs(K - mpmath.sqrt(1 / mpmath.log(2) / mpmath.mpf(0.18)) * 2 ** 61) <= 0.5
    r = np.random.default_rng(5)
    v = r.uniform(-5.6, 5.6, 500) * 2.0 ** r.integers(-130, 1, 500)
    v[:5] = [0.0, -0.0, 5e-324, 5.6, -5.6]
    for x in list(v) + [5.7, 8.0, 11.2]:  # from 2^63 on read as unsigned
        want = mpmath.mpf(float(x)) * K / 4
        got = lib.fx_scale(float(x), K)
        assert abs((got if x < 5.65 else got % 2 ** 64) - want) <= 0.51


@pytest.mark.parametrize("d", [1, 2, 5, 8])
@pytest.mark.parametrize("x,a,b", [((0.5, 5.0), 0.0, 1.0), ((-3.0, 3.0), -1.0, 1.0),
                                   ((1e6, 1e6), 0.0, 1.0), ((1.0, 2.0), 100.0, 101.0),
                                   ((-5.0, -0.5), -2.0, 3.0), ((-1.001, -0.999), 0.9, 1.1)])
def test_poly(lib, d, x, a, b):
    """The root-mean-square error below 2^-52 of g's: a factor is rounded to 2^-60 of its
    largest value and g once to FP64 (2^-54)."""
    r = np.random.default_rng(d)
    n = 400
    xs = r.uniform(x[0], x[1], d)
    v = r.integers(0, 2 ** 23, (n, d), dtype=np.uint32)
    v[0], v[1] = 0, 2 ** 23 - 1
    out = np.empty(n)
    ptr = [z.ctypes.data_as(ctypes.c_void_p) for z in (xs, v, out)]
    assert lib.fx_poly_n(ptr[0], f64(a), f64(b - a), ptr[1], ptr[2], ctypes.c_int(d),
                         ctypes.c_int(n)) == 1
    err, ref = [], []
    for row, g in zip(v, out):
        want = mpmath.mpf(1)
        for xk, vk in zip(xs, row):
            y = mpmath.mpf(a) + mpmath.mpf(b - a) * (2 * int(vk) + 1) / 2 ** 24
            want *= 1 + mpmath.mpf(float(xk)) * y * y
        err.append(float(mpmath.mpf(float(g)) - want))
        ref.append(float(want))
    assert np.sqrt(np.mean(np.square(err)) / np.mean(np.square(ref))) < 2.0 ** -52
    bad = np.full(d, 1e30)
    assert lib.fx_poly_n(bad.ctypes.data_as(ctypes.c_void_p), f64(a), f64(b - a), ptr[1], ptr[2],
                         ctypes.c_int(d), ctypes.c_int(n)) == 0


@pytest.mark.parametrize("n", [1, 2, 1000])
def test_sum(lib, n):
    r = np.random.default_rng(n)
    for g in (r.integers(-2 ** 62, 2 ** 62, n), np.full(n, 2 ** 62), np.full(n, -2 ** 62),
              np.zeros(n, np.int64), np.full(n, 3)):
        g = np.ascontiguousarray(g, np.int64)
        got = lib.fx_sum(g.ctypes.data_as(ctypes.c_void_p), ctypes.c_int(n), ctypes.c_int(62))
        assert got == float(mpmath.mpf(int(sum(int(v) for v in g))) / 2 ** 62)
