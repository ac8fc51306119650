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
