"""Blocks of the pair emission whose ranks touch many super-tiles: all pairs in
the staging area, the pairs of 256 ranks at a time, and pairs of 256 ranks that
exceed it. Against the oracle's lists (integers: no tolerance)."""
import numpy as np
import pytest

from tests.test_gpu_build_chain import _built, _check, _scene  # noqa: F401

pytestmark = pytest.mark.gpu


# one and four ranks per thread (up to 155,648 primitives and more); super-tiles
# counted one by one (up to 1024) and by digits; `wide` Gaussians next to one
# another in depth, `radius` of their distance wide (the staging area holds 4096
# pairs: 256 ranks with more than 16 each exceed it)
@pytest.mark.parametrize("n,wide,radius,size", [(256, 256, 0.05, (512, 512)), (300, 300, 0.1, (1024, 1024)),
                                                (1500, 700, 0.02, (1056, 1024)), (156000, 600, 0.05, (512, 512)),
                                                (156000, 1200, 0.012, (512, 512)), (156000, 300, 0.05, (1056, 1024))])
def test_wide_footprints(orc, n, wide, radius, size):
    sc = _scene(n, n + wide, 0)
    by_depth = np.argsort(sc.means[:, 2])
    at = by_depth[(n - wide) // 2:(n - wide) // 2 + wide]
    sc.scales[at] = (radius * sc.means[at, 2:3]).astype(np.float32)
    _check(orc, sc, orc.gauss_decide, size, 8, "quantile")
