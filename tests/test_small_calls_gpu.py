"""Small calls with host buffers: lists and results go through a pinned buffer, which the
kernels read and write themselves; the results are those of the same scan with device
buffers, bit for bit, at either side of the sizes where the route changes."""
import os
import shutil
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


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


# a cudaHostAlloc that always answers "out of memory" (2), in front of the real one
NO_PINNED = "int cudaHostAlloc(void **p, unsigned long n, unsigned f) { return 2; }\n"
CHILD = """
import ctypes
import numpy as np
from paper_1910_01965_gb300 import zmc
assert ctypes.CDLL(None).cudaHostAlloc(None, ctypes.c_ulong(8), 0) == 2
v = np.linspace(0.5, 5, 20)
mean, err = zmc.zmc_scan(1, 2, [0, 0], [1, 1], [10, 10], v, 1000, 3, 7)
res, _ = zmc.scan(1, 2, [0, 0], [1, 1], [10, 10], v, 1000, 3, 7, want_sums=True)
np.savez(%r, mean=mean, err=err, **{"r_" + k: a for k, a in res.items()})
"""


def test_without_page_locked_memory(zmc, tmp_path):
    """Where no page-locked memory is to be had a small call still runs, by copies."""
    gcc = shutil.which("gcc")
    if not gcc:
        pytest.skip("no gcc")
    (tmp_path / "no.c").write_text(NO_PINNED)
    so, out = str(tmp_path / "no.so"), str(tmp_path / "out.npz")
    subprocess.run([gcc, "-shared", "-fPIC", "-o", so, str(tmp_path / "no.c")], check=True)
    r = subprocess.run([sys.executable, "-c", CHILD % out], cwd=ROOT, capture_output=True,
                       text=True, env=dict(os.environ, LD_PRELOAD=so), timeout=300)
    assert r.returncode == 0, r.stderr[-1500:]
    got = np.load(out)
    v = np.linspace(0.5, 5, 20)
    args = (1, 2, [0, 0], [1, 1], [10, 10], v, 1000, 3, 7)
    mean, err = zmc.zmc_scan(*args)
    res, _ = zmc.scan(*args, want_sums=True)
    assert np.array_equal(got["mean"], mean) and np.array_equal(got["err"], err)
    for k, a in res.items():
        assert np.array_equal(got["r_" + k], a), k
