"""The launch shapes that the planner chooses, from its own functions (no GPU)."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_1910_01965_gb300")
SM = 152


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    from paper_1910_01965_gb300 import zmc
    gxx, cuda = shutil.which("g++"), "/usr/local/cuda/include"
    if not gxx or not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    so = str(tmp_path_factory.mktemp("plan") / "plan.so")
    subprocess.run([gxx, "-O1", "-std=c++17", "-shared", "-fPIC", "-I", os.path.join(PKG, "csrc"),
                    "-I", cuda, "-o", so, os.path.join(ROOT, "tests", "planner_wrap.cpp"),
                    zmc.LIBRARY, "-Wl,-rpath," + os.path.dirname(zmc.LIBRARY)], check=True)
    zmc.load()
    lib = ctypes.CDLL(so)

    def launch_shape(gid, N, T, count, lanes, splits, precision=2, block=256):
        d, keep = zmc.make_desc(gid, N, [0.0] * N, [1.0] * N, [count] + [1] * (N - 1), 0x1000,
                                16384, T, 0, precision, mem=zmc.ZMC_MEM_DEVICE)
        out = (ctypes.c_int * 2)()
        lib.launch_shape(ctypes.byref(d), ctypes.c_int64(count), SM, lanes, splits, block, out)
        return out[0], out[1]

    def batch(scans):
        """(trials, lanes, splits) of each (integrand, N, points, samples, precision)."""
        keep, descs = [], (zmc.zmc_scan_desc * len(scans))()
        for i, (gid, N, points, S, precision) in enumerate(scans):
            d, k = zmc.make_desc(gid, N, [0.0] * N, [1.0] * N, [points] + [1] * (N - 1), 0x1000,
                                 S, 4, 0, precision, mem=zmc.ZMC_MEM_DEVICE)
            keep.append(k)
            descs[i] = d
        counts = (ctypes.c_int64 * len(scans))(*[s[2] for s in scans])
        out = (ctypes.c_int * (3 * len(scans)))()
        lib.batch_trials(descs, counts, len(scans), SM, out)
        return [tuple(out[3 * i:3 * i + 3]) for i in range(len(scans))]

    lib.batch = batch
    lib.shape = launch_shape
    lib.zmc = zmc
    return lib


def test_user_integrands(plan):
    """One trial per lane; blocks of 128 threads only in launches that 256-thread blocks
    would not spread over all SMs."""
    for N in (1, 4, 8):
        for count, block in ((1, 128), (10, 128), (606, 128), (608, 256), (40000, 256)):
            assert plan.shape(plan.zmc.ZMC_G_USER_BASE, N, 8, count, 8, 1) == (1, block)
    assert plan.shape(2, 4, 8, 40000, 4, 1)[0] > 1


@pytest.mark.parametrize("lanes,points", [(128, 2 ** 31 - 2), (128, 2 ** 31 + 2), (32, 2 ** 33),
                                          (128, 2 ** 32 - 4)])
def test_grids_up_to_the_launch_limit(plan, lanes, points):
    """What 256-thread blocks can launch stays launchable: no grid of 2^31 blocks."""
    trials, block = plan.shape(2, 4, 1, points, lanes, 1, precision=0)
    assert points // (block // lanes) <= 2 ** 31 - 1
    assert block == (128 if points * lanes // 128 < 2 ** 31 - 1 else 256)


def test_batches_plan_each_precision_by_itself(plan):
    """A precision's scans share a launch with none of the others, so their plans are
    those of a batch of them alone."""
    fp32 = [(2, 4, 64, 16384, 2)] * 10
    fp64 = [(1, 2, 5000, 65536, 0)] * 40
    plain = [(3, 3, 20000, 16384, 1)] * 5
    alone = plan.batch(fp32) + plan.batch(fp64) + plan.batch(plain)
    assert plan.batch(fp32 + fp64 + plain) == alone
    assert alone[0][0] == 1 and alone[-1][0] > 1  # a short launch and a long one
