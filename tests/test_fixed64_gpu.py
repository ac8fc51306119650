"""FP64 scans whose parameters lie inside, at the edge of and outside the range of the
fixed-point integrands, in one grid, against the oracle."""
import numpy as np
import pytest

import parity
from oracle import oracle
from paper_1910_01965_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

PHASE_X = [0.0, -0.0, 5e-324, -1e-300, 1.7e-5, -3.25, 700.0, 2.0 ** 19, 1048575.5, -2.0 ** 20,
           3e6, 1e9]
BAD_X = [np.inf, -np.inf, np.nan, 1e307]


@pytest.fixture(scope="module")
def zmc():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1910_01965_gb300 import zmc as z
    z.load()
    return z


def _run(z, gid, N, lo, hi, lists, S, T=2, seed=3, tiles=(0, 0, 0)):
    lens = [len(v) for v in lists]
    vals = np.concatenate(lists)
    got, _ = z.scan(gid, N, lo, hi, lens, vals, S, T, seed, precision=z.ZMC_FP64,
                    want_sums=True, tiles=tiles)
    ref = oracle.default().scan(gid, N, lo, hi, lens, vals, S, T, seed, want_sums=True)
    return got, ref


def _compare(got, ref, N, lo, hi, S, phase):
    """1e-12 of scale, plus what FP64 keeps of the phase: the oracle rounds y and
    each product, N 2^-52 of the largest |phase| (one row per grid point).  An error
    d of each g changes sum g^2 by at most 2 d sqrt(S sum g^2) + S d^2, the variance
    that errw is formed from by what the two sums change, and errw by half of that
    over errw, or by its root where errw is smaller."""
    V = float(np.prod(np.asarray(hi) - np.asarray(lo)))
    T = ref["s1"].shape[1]
    d = np.broadcast_to(N * 2.0 ** -52 * phase, ref["mean"].shape)[:, None]
    rms = np.sqrt(ref["s2"] / S)
    tol1 = 1e-12 * S * rms + S * d
    with np.errstate(over="ignore"):
        tol2 = 1e-12 * ref["s2"] + S * d * (2 * rms + d)
    R = V * np.sqrt(np.mean(ref["s2"], axis=1) / S)
    tols = {"s1": tol1, "s2": tol2,
            "mean": 1e-12 * np.maximum(np.abs(ref["mean"]), R) + V * d[:, 0],
            "err": 1e-12 * np.maximum(ref["err"], R) + 2 * V * d[:, 0]}
    if S > 1:
        dvar = np.mean(tol2 + 2 * np.abs(ref["s1"]) / S * tol1, axis=1) / (S - 1)
        tols["errw"] = V * np.sqrt(dvar / (T * S))
        with np.errstate(divide="ignore", invalid="ignore"):
            half = V * V * dvar / (T * S) / (2 * ref["errw"])
        tols["errw"] = 1e-12 * ref["errw"] + np.fmin(tols["errw"], half)
    for name, tol in tols.items():
        ok = np.abs(got[name] - ref[name]) <= tol
        nan = np.isnan(ref[name])
        if name != "errw":  # a negative variance of rounding errors is NaN in one only
            assert np.all(np.isnan(got[name]) == nan), name
        assert np.all(ok | nan | (name == "errw") & np.isnan(got[name])), \
            (name, np.argwhere(~(ok | nan)))


@pytest.mark.parametrize("S,tiles", [(1, (0, 0, 0)), (7, (0, 0, 0)), (1003, (0, 0, 0)),
                                     (1003, (2, 3, 64)), (333, (64, 1, 128))])
@pytest.mark.parametrize("gid", [wl.G_COSPROD, wl.G_OSC01, wl.G_SINSUM])
@pytest.mark.parametrize("N", [1, 2, 5])
def test_phase_ranges(zmc, gid, N, S, tiles):
    x = np.array(PHASE_X + BAD_X)
    lists = [x] + [np.array([0.75])] * (N - 1)
    lo, hi = np.full(N, -1.25), np.full(N, 2.0)
    got, ref = _run(zmc, gid, N, lo, hi, lists, S, tiles=tiles)
    with np.errstate(over="ignore"):
        phase = 2.0 * (np.abs(np.where(np.isfinite(x), x, 0)) + 4 * N)
    _compare(got, ref, N, lo, hi, S, phase)


@pytest.mark.parametrize("lo,hi", [(-1.0, 1.0), (0.0, 1e-9), (1000.0, 1000.5), (-3.0, 8.0),
                                   (1e5, 1e5 + 1), (-2e6, 1.0)])
@pytest.mark.parametrize("gid", [wl.G_COSPROD, wl.G_OSC01, wl.G_SINSUM])
def test_phase_boxes(zmc, gid, lo, hi):
    N, S = 2, 501
    x = np.array([0.5, -2.0, 30.0])
    a, b = np.full(N, lo), np.full(N, hi)
    got, ref = _run(zmc, gid, N, a, b, [x, np.array([1.5])], S)
    m = max(abs(lo), abs(hi))
    quad = 0.1 * m * m if gid == wl.G_OSC01 else 0.0
    _compare(got, ref, N, a, b, S, N * (m * (np.abs(x) + 1.5) + quad))


@pytest.mark.parametrize("N", [1, 3, 5, 8])
@pytest.mark.parametrize("lo,hi", [(-1.0, 1.0), (0.0, 1e-9), (100.0, 101.5), (-5.6, 5.6),
                                   (-30.0, 25.0)])
def test_gauss_ranges(zmc, N, lo, hi):
    """x inside the box, just within and beyond |x - y| = 15.9 / 2.83 and far out (g
    underflows); far from the box the oracle's own exponent is rounded to
    N 2^-53 q nats."""
    mid, half = 0.5 * (lo + hi), 0.5 * (hi - lo)
    x = np.array([mid, lo, hi, mid + 0.3, hi + 5.6 - 2 * half, hi + 5.7, hi + 9.0, hi + 60.0,
                  np.inf, np.nan])
    S, T = 1003, 2
    a, b = np.full(N, lo), np.full(N, hi)
    lists = [x] + [np.array([mid])] * (N - 1)
    got, ref = _run(zmc, wl.G_GAUSS03, N, a, b, lists, S, T)
    V = (hi - lo) ** N
    R = V * np.sqrt(np.mean(ref["s2"], axis=1) / S)
    far = np.maximum(np.abs(x - lo), np.abs(x - hi))
    q = (far ** 2 + (N - 1) * half ** 2) / 0.18
    tol = (1e-12 + N * 2.0 ** -51 * np.where(np.isfinite(q), q, 0)) * \
        np.maximum(np.abs(ref["mean"]), R) + V * 1e-300
    nan = np.isnan(ref["mean"])
    assert np.all(np.isnan(got["mean"]) == nan)
    assert np.all((np.abs(got["mean"] - ref["mean"]) <= tol) | nan)


@pytest.mark.parametrize("N", [1, 2, 3, 5, 8])
@pytest.mark.parametrize("lo,hi", [(0.0, 1.0), (-1.0, 1.0), (100.0, 101.5), (0.0, 1e-9),
                                   (-1e20, 1e20)])
def test_poly_ranges(zmc, N, lo, hi):
    """Factors that change sign, cancel, are tiny, beyond 2^60 and not finite; the
    oracle's rounding of 1 + x y^2 is 3 2^-53 of 1 + |x| y^2 per factor."""
    x = np.array([0.0, 5e-324, -1e-300, 0.7, -0.3, -1.0, 5.0, 1e6, -1e9, 1e30, 1e100, np.inf,
                  np.nan])
    S, T = 1003, 2
    a, b = np.full(N, lo), np.full(N, hi)
    lists = [x] + [np.array([0.6])] * (N - 1)
    with np.errstate(all="ignore"):
        got, ref = _run(zmc, wl.G_POLY, N, a, b, lists, S, T)
        V = (hi - lo) ** N
        y2 = max(abs(lo), abs(hi)) ** 2
        top = (1 + np.abs(x) * y2) * (1 + 0.6 * y2) ** (N - 1)
        R = V * np.sqrt(np.mean(ref["s2"], axis=1) / S)
        tol = 1e-12 * np.fmax(np.abs(ref["mean"]), R) + 4 * N * 2.0 ** -53 * V * top
        same = np.isfinite(ref["mean"]) == np.isfinite(got["mean"])
        ok = np.abs(got["mean"] - ref["mean"]) <= tol
    assert np.all(same)
    assert np.all(ok | ~np.isfinite(ref["mean"]))


def test_unstaged_lists(zmc):
    """More list values than shared memory takes (read from global memory)."""
    r = np.random.default_rng(8)
    x = r.uniform(0.5, 5.0, 5000)
    x[::7] = 3e6
    for gid, lo, hi in ((wl.G_COSPROD, 0.0, 1.0), (wl.G_GAUSS03, -1.0, 1.0)):
        got, ref = _run(zmc, gid, 1, [lo], [hi], [x], 41)
        _compare(got, ref, 1, [lo], [hi], 41, x * (gid == wl.G_COSPROD))


# (integrand, N, parameter, box side) over which |g| is small everywhere: every
# factor near a zero of the cosine, or the phase near a zero of the sine; and next
# to them the bounds' edge, boxes where g is middling.
SMALL_G = [(wl.G_COSPROD, 8, 3.0, 0.5, 0.55), (wl.G_COSPROD, 8, 1.0, 1.5, 1.6),
           (wl.G_COSPROD, 4, 1.0, 1.56, 1.58), (wl.G_COSPROD, 2, 3.14159, 0.499, 0.501),
           (wl.G_COSPROD, 8, 1.5, 1.0, 1.1), (wl.G_COSPROD, 6, 1.5, 1.0, 1.1),
           (wl.G_COSPROD, 3, 1.0, 1.0, 2.0), (wl.G_COSPROD, 8, 1.0, 1.0, 2.0),
           (wl.G_COSPROD, 1, 1.0, 1.5625, 1.578125), (wl.G_COSPROD, 8, 2.25, 0.0, 1.0),
           (wl.G_SINSUM, 1, 0.0, 0.0, 1e-6), (wl.G_SINSUM, 2, 0.0, 0.0, 1e-9),
           (wl.G_SINSUM, 1, 0.0, 0.0, 1e-12), (wl.G_SINSUM, 8, 0.0, -0.01, 0.01),
           (wl.G_SINSUM, 1, 0.0, -0.125, 0.125), (wl.G_SINSUM, 3, 0.0, -1.0, 1.0),
           (wl.G_OSC01, 1, 1.5, 0.979, 0.9835), (wl.G_OSC01, 2, 1.5, 0.506, 0.507),
           (wl.G_OSC01, 1, 0.7927, -4.4, -3.53), (wl.G_OSC01, 3, 1.0, 0.3, 0.7)]


@pytest.mark.parametrize("way", ["scan", "batch", "server"])
@pytest.mark.parametrize("gid,N,x,lo,hi", SMALL_G)
def test_small_integrands(zmc, gid, N, x, lo, hi, way):
    """The sums and the statistics relative to their own size: 1e-12 of sum g^2 and of
    the root mean square, whatever that is (parity.check), in grids that hold an
    ordinary parameter beside the small one (where the box is wide enough for FP64 to
    hold the spread of g that errw is formed from)."""
    S, T = 2003, 3
    lists = [np.array([x, x + (0.4 if hi - lo > 1e-3 else 0.0)])] + [np.array([x])] * (N - 1 if gid != wl.G_SINSUM else 0)
    lens, vals = [len(v) for v in lists], np.concatenate(lists)
    a, b = np.full(N, lo), np.full(N, hi)
    args = (gid, N, a, b, lens, vals, S, T, 5)
    ref = oracle.default().scan(*args, want_sums=True)
    if way == "scan":
        got, _ = zmc.scan(*args, precision=zmc.ZMC_FP64, want_sums=True)
    elif way == "server":
        srv = zmc.Server(1 << 28)
        try:
            t = srv.submit(*args, zmc.ZMC_FP64, want_sums=True)
            assert srv.wait(t, 60000) == zmc.ZMC_OK
            got, _ = srv.result(t)
        finally:
            srv.close()
    else:
        d, keep = zmc.make_desc(*args, zmc.ZMC_FP64)
        got = {"mean": np.empty(2), "err": np.empty(2), "errw": np.empty(2),
               "s1": np.empty((2, T)), "s2": np.empty((2, T))}
        o = zmc.zmc_scan_out()
        for k, v in got.items():
            setattr(o, k, zmc._ptr(v))
        zmc.zmc_scan_batch([d], [o])
    V = float(np.prod(b - a))
    parity.check(got, ref, V, S, 0, way)
    assert np.all(np.abs(got["s2"] - ref["s2"]) <= 1e-12 * ref["s2"])
    assert np.all(np.abs(got["s1"] - ref["s1"]) <= 1e-12 * np.sqrt(S * ref["s2"]))
