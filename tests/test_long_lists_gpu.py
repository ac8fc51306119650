"""FP64 scans, batches and requests whose lists bring a block's shared memory near and
above the 48 KB that a kernel gets without asking (the fixed-point tables take 20, 16
or 36 KB of it), in a process of its own each, in ascending order: a longer list that
ran before would have asked for more already."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SIZES = {"scan": [(1, v) for v in range(3440, 3464)] + [(1, 4096)] +
                 [(2, v) for v in range(3952, 3976)] + [(2, 4096)],
         "batch": [(1, v) for v in range(1396, 1412)] + [(1, 4096)],
         "server": [(1, v) for v in range(1396, 1412)] + [(1, 4096)]}

CHILD = """
import sys
import threading
import numpy as np
from paper_1910_01965_gb300 import zmc

way, sizes = sys.argv[1], eval(sys.argv[2])
r = np.random.default_rng(1)

def args(gid, n):
    return (gid, 1, [0.0], [1.0], [n], r.uniform(0.5, 1.0, n), 40, 2, 7)

def scan(a):
    return zmc.scan(*a, precision=0, count=50)[0]

def batch(a):
    d, keep = zmc.make_desc(*a, 0, count=50)
    res = {k: np.empty(50) for k in ("mean", "err", "errw")}
    o = zmc.zmc_scan_out()
    for k, v in res.items():
        setattr(o, k, zmc._ptr(v))
    zmc.zmc_scan_batch([d], [o])
    return res

server = zmc.Server(1 << 28) if way in ("server", "threads") else None

def serve(a):
    t = server.submit(*a, 0, count=50)
    assert server.wait(t, 60000) == 0, server.wait(t, 0)
    return server.requests.pop(t)[2]

ways = {"scan": scan, "batch": batch, "server": serve}
if way == "threads":
    # one thread each with its own list length, all launching the same kernels
    bad = []
    def work(f, n, times):
        try:
            for _ in range(times):
                f(args(1, n))
        except Exception as e:
            bad.append((n, repr(e)))
    th = [threading.Thread(target=work, args=w)
          for w in ((scan, 3500, 1500), (scan, 4000, 1500), (batch, 1500, 300), (serve, 4000, 300),
                    (batch, 3000, 300))]
    [t.start() for t in th]
    [t.join() for t in th]
    assert not bad, bad
else:
    for gid, n in sizes:
        a = args(gid, n)
        got = ways[way](a)
        few = zmc.scan(gid, 1, [0.0], [1.0], [50], a[5][:50], 40, 2, 7, precision=0)[0]
        assert np.allclose(got["mean"], few["mean"], rtol=1e-13, atol=0), (gid, n)
if server:
    server.close()
print("done")
"""


@pytest.mark.parametrize("way", ["scan", "batch", "server", "threads"])
def test_shared_memory_limit(way):
    r = subprocess.run([sys.executable, "-c", CHILD, way, repr(SIZES.get(way))], cwd=ROOT,
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "done" in r.stdout, r.stderr[-1500:]
