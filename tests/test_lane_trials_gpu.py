"""Lanes that sample several trials of a point together (4, 2 or 1, and blocks that
mix them).  A trial's sums do not depend on how many trials a scan has, so scans of
1 to 8 trials are compared bit for bit on the trials they share."""
import numpy as np
import pytest

from paper_1910_01965_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

GIDS = [wl.G_COSPROD, wl.G_GAUSS03, wl.G_POLY, wl.G_OSC01, wl.G_SINSUM, wl.G_CONST]


@pytest.fixture(scope="module")
def zmc():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1910_01965_gb300 import zmc as z
    z.load()
    return z


@pytest.mark.parametrize("prec", [1, 2, 0])
@pytest.mark.parametrize("N", [1, 2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("tiles", [(1, 1, 64), (4, 2, 256), (32, 1, 128), (64, 3, 256),
                                   (512, 1, 512)])
def test_trials_do_not_depend_on_their_company(zmc, prec, N, tiles):
    """T = 1 to 8, with enough points that the lanes of the larger ones take several
    trials and blocks hold the borders between lane groups of four, two and one."""
    r = np.random.default_rng(N)
    gid = GIDS[N % 6]
    S = 83 + N
    # enough blocks for several rounds on any SM count, whatever the lanes
    points = 40 * 200 * max(1, tiles[2] // tiles[0]) // (4 * tiles[1]) if tiles[0] < 64 else 700
    lens = [points] + [1] * (N - 1)
    vals = r.uniform(0.2, 1.5, points + N - 1)
    args = (gid, N, [0.0] * N, [1.0] * N, lens, vals, S)
    base = None
    for T in (8, 7, 5, 4, 3, 2, 1):
        res, o = zmc.scan(*args, T, 11, precision=prec, tiles=tiles, want_sums=True)
        if base is None:
            base = res
        assert np.array_equal(res["s1"], base["s1"][:, :T]), T
        assert np.array_equal(res["s2"], base["s2"][:, :T]), T


@pytest.mark.parametrize("points,S,scans", [(1, 1, 1), (3, 1003, 5), (700, 4001, 3),
                                            (6000, 3001, 40)])
def test_batches_of_all_sizes_equal_solo_runs(zmc, points, S, scans):
    """From a few lanes (short lanes, one trial each) to many rounds of tiles (lanes of
    four trials): each scan of a batch equals its solo run with the batch's tiles."""
    import torch
    r = np.random.default_rng(scans)
    descs, outs, keep, want = [], [], [], []
    for i in range(scans):
        N, T, prec = 1 + i % 8, (4, 5, 7, 1, 2)[i % 5], (2, 1, 0)[i % 3]
        lens = [points] + [1] * (N - 1)
        vals = r.uniform(0.2, 1.5, points + N - 1)
        args = (GIDS[i % 6], N, [0.0] * N, [1.0] * N, lens, vals, S, T, 5 + i)
        v = torch.from_numpy(vals).cuda()
        d, k = zmc.make_desc(*args[:5], v, S, T, 5 + i, prec, zmc.ZMC_MEM_DEVICE)
        res = [torch.empty(points, dtype=torch.float64, device="cuda") for _ in range(2)] + \
            [torch.empty((points, T), dtype=torch.float64, device="cuda") for _ in range(2)]
        o = zmc.zmc_scan_out()
        o.mean, o.err, o.s1, o.s2 = (zmc._ptr(x) for x in res)
        descs.append(d)
        outs.append(o)
        keep.append((v, k, res))
        want.append((args, prec))
    h = zmc.zmc_batch_create(descs, outs)
    zmc.zmc_batch_run(h)
    torch.cuda.synchronize()
    for (args, prec), o, (_, _, res) in zip(want, outs, keep):
        solo, _ = zmc.scan(*args, precision=prec, want_sums=True,
                           tiles=(o.tile_lanes, o.tile_splits, o.tile_block))
        assert np.array_equal(solo["s1"], res[2].cpu().numpy())
        assert np.array_equal(solo["s2"], res[3].cpu().numpy())
    zmc.zmc_batch_destroy(h)


def test_server_budget_takes_the_longest_lanes(zmc):
    """A request whose partial sums exceed the budget with short lanes (1 MB here, with
    0.6 MB of lists and results) is planned with the longest ones and served."""
    P, T, S = 2000, 8, 1 << 17
    vals = np.linspace(0.5, 5.0, P)
    args = (wl.G_COSPROD, 1, [0.0], [1.0], [P], vals, S, T, 3)
    srv = zmc.Server(1 << 20)
    try:
        t = srv.submit(*args, want_sums=True)
        assert srv.wait(t) == zmc.ZMC_OK
        res, o = srv.result(t)
        solo, _ = zmc.scan(*args, want_sums=True,
                           tiles=(o.tile_lanes, o.tile_splits, o.tile_block))
        assert np.array_equal(res["s1"], solo["s1"])
        assert np.array_equal(res["mean"], solo["mean"])
    finally:
        srv.close()
