"""Small calls with host buffers: lists and results go through a pinned buffer, which the
kernels read and write themselves; the results are those of the same scan with device
buffers, bit for bit, at either side of the sizes where the route changes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def zmc():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1910_01965_gb300 import zmc as z
    z.load()
    return z


# list values, points: lists read in place up to 256 and above 4096 values, calls of at
# most 2^18 bytes of lists and results
SIZES = [(20, 1), (20, 100), (255, 700), (256, 700), (257, 700), (1024, 700), (4096, 700),
         (4097, 700), (12000, 6000), (2768, 4000), (4768, 4000), (4769, 4000), (60, 4672), (60, 4673)]


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("nvals,count", SIZES)
def test_host_equals_device(zmc, nvals, count, prec):
    import torch
    r = np.random.default_rng(nvals)
    N = 2
    while (nvals // N) ** N < count:  # more lists, until the grid is large enough
        N += 1
    lens = [nvals - (N - 1) * (nvals // N)] + [nvals // N] * (N - 1)
    N = len(lens)
    vals = r.uniform(0.5, 3.0, nvals)
    args = (1, N, [0.0] * N, [1.0] * N, lens)
    rest = (203, 2, 9)
    got, _ = zmc.scan(*args, vals, *rest, precision=prec, count=count, want_sums=True)
    dev = {k: torch.empty(count * (2 if k in ("s1", "s2") else 1), dtype=torch.float64,
                          device="cuda") for k in got}
    zmc.scan_device(*args, torch.from_numpy(vals).cuda(), *rest, precision=prec, count=count,
                    **{"out_" + k: v for k, v in dev.items()})
    torch.cuda.synchronize()
    for k in got:
        assert np.array_equal(got[k].ravel(), dev[k].cpu().numpy()), k
