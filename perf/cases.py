"""Performance cases: the scans, batches and served requests that programs make.

A case names the integrand, its dimension N, the lengths of the parameter lists,
samples per point S, trials T, the precision and the way in:

  host    zmc.scan: lists and results in host memory, one synchronous call
  simple  zmc.zmc_scan: the seven-argument host call (FP32 with Kahan sums)
  device  zmc.scan_device: lists and results in device memory, enqueued on the
          current stream; optionally a slice of the grid and the per-trial sums
  batch   zmc_batch_run of a prepared batch of uneven scans (one captured graph)
  server  a burst of requests submitted to a running server, all waited for

Boxes and parameter ranges follow the repository's workloads: cos-product and
polynomial on [0,1]^N with x ~ U[0.5, 5], Gaussian on [-1,1]^N with x ~ U[-1, 1],
oscillatory on [0,2]^N with x ~ U[0.5, 5], sine-sum on [0,1]^N with x in {0..99}.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_1910_01965_gb300 import zmc

GIDS = {"cosprod": zmc.ZMC_G_COSPROD, "gauss": zmc.ZMC_G_GAUSS03, "poly": zmc.ZMC_G_POLY,
        "osc": zmc.ZMC_G_OSC01, "sinsum": zmc.ZMC_G_SINSUM}
BOX = {"cosprod": (0.0, 1.0), "gauss": (-1.0, 1.0), "poly": (0.0, 1.0), "osc": (0.0, 2.0),
       "sinsum": (0.0, 1.0)}

# Largest number of uniforms (samples x dimensions) that exact() recomputes.
EXACT_FIELDS = 2.0e10


def listed():
    return [
        # The first call of the README: a 10 x 10 grid from host lists, latency above all.
        dict(name="quickstart_cosprod_100", kind="simple", g="cosprod", N=2, lens="10,10",
             S=65536, T=5, prec="fp32_kahan"),
        # The same grid in FP64 with all three statistics: the parity workload.
        dict(name="cosprod_100_fp64", kind="host", g="cosprod", N=2, lens="10,10",
             S=65536, T=5, prec="fp64"),
        # A small odd-sized call with few samples, as a fitting loop makes it.
        dict(name="poly_small_odd", kind="host", g="poly", N=3, lens="7,11,3", S=1003, T=3,
             prec="fp32_kahan"),
        # The headline scan: 10^6 points in device memory.
        dict(name="gauss_1e6", kind="device", g="gauss", N=4, lens="100,100,100,1", S=16384,
             T=4, prec="fp32_kahan"),
        # The sine-sum test of the paper, one trial per point, host buffers.
        dict(name="sinsum_grid3", kind="host", g="sinsum", N=4, lens="100,100,60", S=10000,
             T=1, prec="fp32_kahan"),
        # Precision stress: oscillatory in six dimensions, many samples, eight trials.
        dict(name="osc_1e4", kind="device", g="osc", N=6, lens="10,10,10,10,1,1", S=32768,
             T=8, prec="fp32_kahan"),
        # The FP64 path on a grid that fills the GPU: Gaussian in four dimensions.
        dict(name="gauss_fp64", kind="device", g="gauss", N=4, lens="25,20,20,1", S=4096, T=4,
             prec="fp64"),
        # The FP64 path on the oscillatory integrand, ragged sample count.
        dict(name="osc_fp64", kind="device", g="osc", N=6, lens="10,10,9,1,1,1", S=20011, T=5,
             prec="fp64"),
        # Plain FP32 sums, seven dimensions, odd sizes, a slice of the grid (one
        # rank's or one checkpoint's share) with its per-trial sums.
        dict(name="poly_fp32_slice", kind="device", g="poly", N=7, lens="33,31,29,1,1,1,1",
             S=10007, T=4, prec="fp32", first=1001, count=24571, sums=True),
        # A large grid streamed to host memory in chunks, few samples per point.
        dict(name="cosprod_stream", kind="host", g="cosprod", N=3, lens="151,149,139", S=1024,
             T=4, prec="fp32_kahan"),
        # Uneven scans in one persistent launch, replayed as a graph.
        dict(name="batch_uneven_64", kind="batch", mix=1, scans=64, pmax=20000, smax=65536,
             T=4, prec="fp32_kahan"),
        # A burst of small requests to a running server.
        dict(name="server_burst_48", kind="server", mix=2, scans=48, pmax=3000, smax=16384,
             T=4, prec="fp32_kahan"),
    ]


def _logint(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    kind = rng.choice(["simple", "host", "device", "device", "host", "batch", "server"])
    if kind in ("batch", "server"):
        return dict(kind=kind, mix=rng.randrange(3, 1 << 20), scans=_logint(rng, 8, 64),
                    pmax=_logint(rng, 100, 6000), smax=_logint(rng, 4096, 32768), T=4,
                    prec="fp32_kahan")
    g = rng.choice(sorted(GIDS))
    N = rng.randrange(1, 9)
    prec = "fp32_kahan" if kind == "simple" else \
        rng.choice(["fp32_kahan", "fp32_kahan", "fp64", "fp32"])
    T = rng.choice([1, 2, 3, 4, 4, 5, 8])
    S = _logint(rng, 500, 200000)
    # evaluations bounded by the dearest of the listed cases of that precision
    budget = (1.2e9 if prec == "fp64" else 2.0e10) / N / (S * T)
    P = min(_logint(rng, 10, 1e6), max(1, int(budget)))
    m = min(N, 3) if g != "sinsum" else rng.randrange(1, 5)
    side = max(1, int(round(P ** (1.0 / m))))
    lens = [side] * m
    lens[-1] = max(1, P // side ** (m - 1))
    if g != "sinsum":
        lens += [1] * (N - m)
    return dict(kind=kind, g=g, N=N, lens=",".join(str(v) for v in lens), S=S, T=T, prec=prec)


def _mix(case):
    """The scans of a batch or a burst: their sizes belong to the case, not to the seed."""
    rng = random.Random(case["mix"])
    out = []
    for i in range(case["scans"]):
        N = rng.randrange(1, 9)
        P = _logint(rng, 10, case["pmax"])
        S = max(4, int(round(_logint(rng, 1024, case["smax"]) / 4.0)) * 4)
        m = min(N, 3)
        lens = [max(1, int(round(P ** (1.0 / m))))] * m + [1] * (N - m)
        out.append(dict(g=rng.choice(["cosprod", "gauss", "poly"]), N=N,
                        lens=",".join(str(v) for v in lens), S=S, T=case["T"],
                        prec=case["prec"]))
    return out


def _spec(c, seed, index=0):
    """One scan's inputs: (gid, N, lo, hi, lens, list values, S, T, Philox seed)."""
    rng = np.random.default_rng([int(seed), index])
    lens = [int(v) for v in c["lens"].split(",")]
    g, N = c["g"], c["N"]
    lists = []
    for L in lens:
        if g == "gauss":
            lists.append(rng.uniform(-1.0, 1.0, L))
        elif g == "sinsum":
            lists.append(rng.integers(0, 100, L).astype(np.float64))
        else:
            lists.append(rng.uniform(0.5, 5.0, L))
    a, b = BOX[g]
    key = (int(seed) * 0x9E3779B97F4A7C15 + index * 0xD1B54A32D192ED03 + 1) & (2 ** 64 - 1)
    return (GIDS[g], N, np.full(N, a), np.full(N, b), np.array(lens, np.int64),
            np.concatenate(lists), c["S"], c["T"], key)


def _count(c):
    P = int(np.prod([int(v) for v in c["lens"].split(",")]))
    return c.get("count", P)


class _Batch:
    """A prepared batch: descriptors, device buffers and the library's handle."""

    def __init__(self, scans, seed):
        # one device array per statistic; each scan writes its own stretch
        total = sum(_count(c) for c in scans)
        self.outs = [torch.empty(total, dtype=torch.float64, device="cuda") for _ in range(3)]
        self.keep, descs, outs, at = [], [], [], 0
        for i, c in enumerate(scans):
            gid, N, lo, hi, lens, vals, S, T, key = _spec(c, seed, i)
            v = torch.from_numpy(vals).cuda()
            d, keep = zmc.make_desc(gid, N, lo, hi, lens, v, S, T, key,
                                    zmc.PRECISIONS[c["prec"]], zmc.ZMC_MEM_DEVICE)
            o = zmc.zmc_scan_out()
            o.mean, o.err, o.errw = (zmc._ptr(r[at:at + _count(c)]) for r in self.outs)
            at += _count(c)
            self.keep.append((keep, v))
            descs.append(d)
            outs.append(o)
        torch.cuda.synchronize()
        self.handle = zmc.zmc_batch_create(descs, outs, zmc.ZMC_BATCH_GRAPH)

    def __del__(self):
        if getattr(self, "handle", None):
            zmc.zmc_batch_destroy(self.handle)


class _Server(zmc.Server):
    def __del__(self):
        if getattr(self, "handle", None):
            self.close()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return ("batch", _Batch(_mix(case), seed))
    if kind == "server":
        return ("server", _Server(4 << 30), [_spec(c, seed, i) for i, c in enumerate(_mix(case))])
    spec = _spec(case, seed)
    prec = zmc.PRECISIONS[case["prec"]]
    if kind == "device":
        n, T = _count(case), case["T"]
        bufs = {k: torch.empty(n, dtype=torch.float64, device="cuda")
                for k in ("out_mean", "out_err", "out_errw")}
        if case.get("sums"):
            bufs.update({k: torch.empty((n, T), dtype=torch.float64, device="cuda")
                         for k in ("out_s1", "out_s2")})
        vals = torch.from_numpy(spec[5]).cuda()
        kw = dict(precision=prec, first_index=case.get("first", 0), count=case.get("count", -1))
        return ("device", spec[:5] + (vals,) + spec[6:], bufs, kw)
    return (kind, spec, prec)


def run(state):
    kind = state[0]
    if kind == "simple":
        return list(zmc.zmc_scan(*state[1]))
    if kind == "host":
        res, _ = zmc.scan(*state[1], precision=state[2])
        return [res["mean"], res["err"], res["errw"]]
    if kind == "device":
        zmc.scan_device(*state[1], stream=torch.cuda.current_stream().cuda_stream, **state[2],
                        **state[3])
        return list(state[2].values())
    if kind == "batch":
        zmc.zmc_batch_run(state[1].handle, torch.cuda.current_stream().cuda_stream)
        return state[1].outs
    server, specs = state[1], state[2]
    tickets = [server.submit(*s) for s in specs]
    outs = []
    for t in tickets:
        status = server.wait(t)
        if status != zmc.ZMC_OK:
            raise RuntimeError("request ended with %s" % zmc.STATUS_NAMES[status])
        res, _ = server.result(t)
        outs.append((res["mean"], res["err"], res["errw"]))
        server.requests.pop(t)
    return [np.concatenate(v) for v in zip(*outs)]


def _scans(case):
    return _mix(case) if case["kind"] in ("batch", "server") else [case]


def work(case):
    """Bytes: the lists in, the results out.  Operations per evaluation: 8 N for the
    counter-based generator (40 per call of five uniforms), 2 N for the map into the
    box, the integrand's own and the two sums'."""
    own = {"cosprod": lambda N: 3 * N - 1, "gauss": lambda N: 2 * N + 2,
           "poly": lambda N: 3 * N - 1, "osc": lambda N: 2 * N + 2, "sinsum": lambda N: N + 2}
    nbytes = flops = 0
    for c in _scans(case):
        n = _count(c)
        per = 8 * c["N"] + 2 * c["N"] + own[c["g"]](c["N"]) + \
            (9 if c["prec"] == "fp32_kahan" else 2)
        stats = 2 if case["kind"] == "simple" else 3
        nbytes += 8 * sum(int(v) for v in c["lens"].split(",")) + 8 * n * stats
        if c.get("sums"):
            nbytes += 16 * n * c["T"]
        flops += n * c["T"] * c["S"] * per
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """About four times the largest deviation of any output from exact() that was
    measured, by precision and integrand, over the listed cases and 76 drawn ones:
    FP64 1.3e-14 (err, the spread of the trial means, which magnifies rounding);
    FP32 5.9e-5 for the oscillatory integrand (its mean over many dimensions is near
    zero), 2.3e-6 for the sine-sum, 9e-7 for the others, 9.2e-6 with plain FP32 sums
    (err again), 1.3e-7 for mixes."""
    if case["prec"] == "fp64":
        return {"rel": 6e-14}
    if "mix" in case:
        return {"rel": 6e-7}
    rel = {"osc": 2.5e-4, "sinsum": 1e-5}.get(case["g"], 4e-6)
    return {"rel": max(rel, 4e-5) if case["prec"] == "fp32" else rel}


# ------------------------------------------------------------------- exact --
def _philox_fields(seed, p, T, first_call, ncalls, dev):
    """The five 23-bit fields of `ncalls` Philox4x32-10 calls for each (point, trial):
    int64 [points, T, ncalls, 5]."""
    M32 = 0xFFFFFFFF
    j = torch.arange(first_call, first_call + ncalls, device=dev, dtype=torch.int64)
    x0 = j.view(1, 1, -1)
    x1 = torch.arange(T, device=dev, dtype=torch.int64).view(1, -1, 1)
    x2 = (p & M32).view(-1, 1, 1)
    x3 = (p >> 32).view(-1, 1, 1)
    k0, k1 = seed & M32, (seed >> 32) & M32
    for _ in range(10):
        a = x0 * 0xD2511F53
        b = x2 * 0xCD9E8D57
        x0, x1, x2, x3 = (((b >> 32) & M32) ^ x1 ^ k0, b & M32, ((a >> 32) & M32) ^ x3 ^ k1,
                          a & M32)
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    r = torch.broadcast_tensors(x0, x1, x2, x3)
    m = 0x7FFFFF
    return torch.stack([r[0] & m, (r[0] >> 23 | r[1] << 9) & m, (r[1] >> 14 | r[2] << 18) & m,
                        (r[2] >> 5) & m, (r[2] >> 28 | r[3] << 4) & m], dim=-1)


def _g64(name, y, x):
    """The integrand at y [points, T, samples, N] for x [points, M], in 64 bits."""
    N = y.shape[-1]
    xs = x[:, :N].view(x.shape[0], 1, 1, -1)
    if name == "cosprod":
        return torch.cos(xs * y).prod(dim=-1)
    if name == "gauss":
        return torch.exp(-((y - xs) ** 2).sum(dim=-1) / (2 * 0.3 ** 2))
    if name == "poly":
        return (1 + xs * y * y).prod(dim=-1)
    if name == "osc":
        return torch.cos((xs * y + 0.1 * y * y).sum(dim=-1))
    return torch.sin(y.sum(dim=-1) + x.sum(dim=1).view(-1, 1, 1))


def _exact_scan(c, seed, index, dev):
    gid, N, lo, hi, lens, vals, S, T, key = _spec(c, seed, index)
    first, n = c.get("first", 0), _count(c)
    lists = [torch.from_numpy(v).to(dev) for v in np.split(vals, np.cumsum(lens)[:-1])]
    a, w = float(lo[0]), float(hi[0] - lo[0])
    s1 = torch.zeros((n, T), dtype=torch.float64, device=dev)
    s2 = torch.zeros_like(s1)
    limit = 1 << 25                          # uniforms held at a time
    sblk = min(S, max(5, limit // (T * N) // 5 * 5))   # whole calls: 5 | sblk
    pblk = max(1, limit // (sblk * T * N))
    for p0 in range(0, n, pblk):
        p = torch.arange(first + p0, first + min(n, p0 + pblk), device=dev, dtype=torch.int64)
        q, cols = p, [None] * len(lens)
        for i in range(len(lens) - 1, -1, -1):
            cols[i] = lists[i][q % int(lens[i])]
            q = torch.div(q, int(lens[i]), rounding_mode="floor")
        x = torch.stack(cols, dim=1)
        for s0 in range(0, S, sblk):
            m = min(sblk, S - s0)
            f = _philox_fields(key, p, T, s0 * N // 5, -(-m * N // 5), dev)
            f = f.view(len(p), T, -1)[:, :, :m * N].reshape(len(p), T, m, N)
            y = a + w * ((2 * f + 1).to(torch.float64) * 2.0 ** -24)
            g = _g64(c["g"], y, x)
            s1[p0:p0 + len(p)] += g.sum(dim=-1)
            s2[p0:p0 + len(p)] += (g * g).sum(dim=-1)
    V = w ** N
    I = V * s1 / S
    mean = I.mean(dim=1)
    nan = torch.full_like(mean, float("nan"))
    err = (((I - mean[:, None]) ** 2).sum(dim=1) / (T * (T - 1))).sqrt() if T > 1 else nan
    errw = V * (((s2 - s1 * s1 / S) / (S - 1)).mean(dim=1) / (T * S)).sqrt() if S > 1 else nan
    return mean, err, errw, s1, s2


def exact(case, seed):
    scans = _scans(case)
    if sum(_count(c) * c["T"] * c["S"] * c["N"] for c in scans) > EXACT_FIELDS:
        return None
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    keep = 2 if case["kind"] == "simple" else 5 if case.get("sums") else 3
    out = []
    for i, c in enumerate(scans):
        out.append([t.cpu().numpy() for t in _exact_scan(c, seed, i, dev)[:keep]])
    return [np.concatenate(v) for v in zip(*out)]
