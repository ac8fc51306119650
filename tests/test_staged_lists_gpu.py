"""Lists staged into shared memory four values at a time (one dimension) against the
unstaged list, at the remainders of the groups of values."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gid", [1, 2, 3, 4])
@pytest.mark.parametrize("block", [64, 128, 256])
def test_lengths(gid, block):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1910_01965_gb300 import zmc
    vals = np.random.default_rng(gid).uniform(0.5, 3.0, 4097)
    tiles = (8, 1, block)

    def run(n):
        # the first points of the grid: their streams do not depend on the list's length
        return zmc.scan(gid, 1, [0.0], [1.0], [n], vals[:n], 200, 2, 7, tiles=tiles)[0]

    whole = run(4097)  # not staged
    for n in (1, 2, block - 1, block, block + 1, 3 * block, 4 * block - 1, 4 * block,
              4 * block + 1, 7 * block + 5, 4095, 4096):
        got = run(n)
        for k in got:
            assert np.array_equal(got[k], whole[k][:n]), (n, k)
