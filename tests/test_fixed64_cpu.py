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


@pytest.mark.parametrize("scale", [60, 62])
def test_square(lib, scale):
    """g^2 to two units of 2^-scale, without a bias that grows with the sum."""
    r = np.random.default_rng(6)
    g = np.concatenate([r.integers(-2 ** 62, 2 ** 62, 4000), r.integers(-2 ** 50, 2 ** 50, 100),
                        [2 ** 62, -2 ** 62, 0, 1, -1]])
    got = _call(lib.fx_square_60 if scale == 60 else lib.fx_square_62, np.int64, len(g), g)
    err = np.array([float(mpmath.mpf(int(q)) - mpmath.mpf(int(v)) ** 2 / 2 ** (124 - scale))
                    for q, v in zip(got, g)])
    assert np.max(np.abs(err)) <= 2.0
    assert abs(err[:4000].mean()) < 5 * err[:4000].std() / np.sqrt(4000) + 0.4


LD = np.longdouble


def _cosprod(lib, d, x, a, w, v):
    n = len(v)
    m, least = np.zeros(1, np.float32), np.zeros(1, np.float32)
    g, sq = np.empty(n, np.int64), np.empty(n, np.int64)
    ptr = [z.ctypes.data_as(ctypes.c_void_p) for z in (x, v, m, least, g, sq)]
    lib.fx_cosprod_n(ptr[0], f64(a), f64(w), ptr[1], d, n, *ptr[2:])
    ok = least[0] >= 2.0 ** -6 and m[0] >= (2.0 ** -8 if d <= 5 else 2.0 ** -11)
    return ok, float(m[0]), g, sq, 60 if d <= 3 else 62


def _sinsum(lib, d, xsum, a, w, v):
    n = len(v)
    m, g, sq = np.zeros(1, np.float32), np.empty(n, np.int64), np.empty(n, np.int64)
    ptr = [z.ctypes.data_as(ctypes.c_void_p) for z in (a, w, v, m, g, sq)]
    lib.fx_sinsum_n(f64(xsum), *ptr[:3], d, n, *ptr[3:])
    return m[0] >= 2.0 ** -6, float(m[0]), g, sq, 60


def _errors(g, sq, scale, ex, n):
    """Root-mean-square errors of g and of g^2 over R and R^2."""
    R2 = np.mean(ex ** 2)
    e1 = np.mean((g.astype(LD) * LD(2) ** -62 - ex) ** 2) / R2
    e2 = np.mean((sq.astype(LD) * LD(2) ** -scale - ex ** 2) ** 2) / R2 ** 2
    return float(np.sqrt(e1)), float(np.sqrt(e2)), float(R2)


def test_range_of_small_cosines(lib):
    """Boxes that the range tests let through, most of them near the line: the errors
    of g below 2^-53 R and of g^2 below 2^-50 R^2 (one FP64 rounding is 2^-54.8 of a
    value); the estimate of R^2 agrees with the samples' within their spread; and boxes
    over which every factor is small, however many, are out."""
    r = np.random.default_rng(7)
    near = 0
    for t in range(400):
        d = int(r.integers(1, 9))
        x = r.uniform(0.5, 5.0, d) if t % 4 == 0 else np.full(d, r.uniform(0.5, 5.0))
        w = float(10 ** r.uniform(-2, 0.5))
        a = float(r.uniform(-2, 2) if t % 4 == 0 else np.pi / 2 / x[0] - w * r.uniform())
        v = r.integers(0, 2 ** 23, (500, d), dtype=np.uint32)
        ok, m, g, sq, scale = _cosprod(lib, d, x, a, w, v)
        y = LD(a) + LD(w) * (2 * v.astype(LD) + 1) * LD(2) ** -24
        ex = np.cos(x.astype(LD) * y).prod(axis=1)
        e1, e2, R2 = _errors(g, sq, scale, ex, len(v))
        assert abs(m - R2) < 6 * float(np.std(ex ** 2)) / np.sqrt(500) + 1e-5, (d, x, a, w)
        if ok:
            near += m < 2.0 ** -6
            assert e1 < 2.0 ** -53 and e2 < 2.0 ** -50, (d, x, a, w)
    assert near > 20
    for d, x, a, w in ((8, 3.0, 0.5, 0.05), (8, 1.0, 1.5, 0.1), (4, 1.0, 1.56, 0.02),
                       (2, 3.14159, 0.499, 0.002), (6, 1.5, 1.0, 0.1), (8, 1.0, 1.0, 1.0)):
        assert not _cosprod(lib, d, np.full(d, x), a, w, np.zeros((1, d), np.uint32))[0]


def test_range_of_small_sines(lib):
    r = np.random.default_rng(8)
    for t in range(400):
        d = int(r.integers(1, 9))
        w, a = 10 ** r.uniform(-2, 0.3, d), r.uniform(-1, 1, d)
        xsum = float(-a.sum() - w.sum() * r.uniform()) if t % 2 else float(r.integers(0, 400))
        v = r.integers(0, 2 ** 23, (500, d), dtype=np.uint32)
        ok, m, g, sq, scale = _sinsum(lib, d, xsum, a, w, v)
        y = a.astype(LD) + w.astype(LD) * (2 * v.astype(LD) + 1) * LD(2) ** -24
        ex = np.sin(y.sum(axis=1) + LD(xsum))
        e1, e2, R2 = _errors(g, sq, scale, ex, len(v))
        assert abs(m - R2) < 6 * float(np.std(ex ** 2)) / np.sqrt(500) + 1e-5
        assert not ok or (e1 < 2.0 ** -53 and e2 < 2.0 ** -50)
    for w in (1e-12, 1e-6, 0.2):
        assert not _sinsum(lib, 1, 0.0, np.zeros(1), np.full(1, w), np.zeros((1, 1), np.uint32))[0]


def test_range_of_oscillatory_phases(lib):
    """The reach of x y + 0.1 y^2 against a fine grid, and |cos| over a stretch of
    phases against its least there."""
    r = np.random.default_rng(9)
    out = np.empty(2, np.float32)
    f32 = ctypes.c_float
    for t in range(300):
        x, a, w = r.uniform(-2, 2), r.uniform(-10, 10), 10 ** r.uniform(-2, 1)
        if t % 2:
            x = -0.2 * (a + w * r.uniform())  # lowest inside the box
        lib.fx_quad(f32(x), f32(0.1), f32(a), f32(w), out.ctypes.data_as(ctypes.c_void_p))
        y = a + w * np.linspace(0, 1, 20001)
        p = x * y + 0.1 * y * y
        size = abs(x) * w + 0.2 * (abs(a) + w) * w
        assert abs(out[0] - np.ptp(p)) < 1e-5 * size and abs(out[1] - (p[0] - p.min())) < 1e-5 * size
        start, width = r.uniform(0, 1), r.uniform(0, 1.2)
        least = np.abs(np.cos(2 * np.pi * start + width * np.linspace(0, 1, 2001))).min()
        got = lib.fx_range(u32(int(start * 2 ** 32)), f32(width))
        if width >= 1.0:
            assert got
        elif abs(least - 0.25) > 1e-3:
            assert bool(got) == (least > 0.25), (start, width)
