"""The build up to the tile lists (culling, depth order, planes, lists) against
the FP64 oracle at the edges of its kernels, on scenes that are too large for
the oracle's splats. Everything here is integers or FP64 bits: no tolerance."""
import numpy as np
import pytest
import torch

from paper_2508_18540_gb300 import api
from paper_2508_18540_gb300 import synth as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2508_18540_gb300 import build
    build.build()


def _scene(n, seed, ties):
    """Small Gaussians all over the frustum; ties > 0 rounds the depths to
    that many values, so equal keys come in runs."""
    rng = np.random.default_rng(seed)
    z = rng.uniform(1.0, 9.0, n)
    if ties:
        z = 1.0 + np.floor((z - 1.0) / 8.0 * ties) / ties * 8.0
    xy = rng.uniform(-0.5, 0.5, (n, 2)) * z[:, None]
    f = np.float32
    q = rng.normal(size=(n, 4))
    return S.GaussianScene(np.column_stack([xy, z]).astype(f), np.full((n, 3), 0.002, f), q.astype(f),
                           np.full(n, 0.5, f), np.full((n, 3), 0.5, f))


def _lists(o, W, H, N):
    """All (tile, plane) lists as one array of indices and their start offsets."""
    tiles_x, tiles_y = (W + 15) // 16, (H + 15) // 16
    g = o["order"]
    t = o["rect"][g] // 16
    nx, ny = t[:, 2] - t[:, 0] + 1, t[:, 3] - t[:, 1] + 1
    rep = np.repeat(np.arange(len(g)), nx * ny)
    k = np.arange(len(rep)) - np.repeat(np.cumsum(nx * ny) - nx * ny, nx * ny)
    tile = (t[rep, 1] + k // nx[rep]) * tiles_x + t[rep, 0] + k % nx[rep]
    seg = tile.astype(np.int64) * N + o["chunk"][g][rep]
    by = np.argsort(seg, kind="stable")                 # keeps the depth order
    return g[rep][by], np.concatenate([[0], np.cumsum(np.bincount(seg, minlength=tiles_x * tiles_y * N))])


def _check(orc, scene, decide, size, N, binning, dtype="f16"):
    W, H = size
    cam = S.Camera(np.eye(3), np.zeros(3), np.radians(50.0), np.radians(50.0), W, H)
    disp = S.display_for(3.0, 0.1)
    ref = orc.make_ref(cam, disp)
    z, valid, rect = decide(ref, scene)
    order, chunk, d, count, M = orc.bin_primitives(ref, z, valid, N, binning)
    r = api.LightFieldRenderer(cam, disp, S.ViewSet(1, 1), N, binning, dtype)
    prims = api.DeviceVoxels.from_scene(scene) if hasattr(scene, "ijk") else api.DeviceGaussians.from_scene(scene)
    pl = r.build(prims)
    st, _, gm = r.status()
    assert st == 0 and gm == M
    n = scene.n
    assert np.array_equal(pl.rect[:n].cpu().numpy(), rect)
    assert np.array_equal(pl.chunk[:n].cpu().numpy(), chunk)
    assert np.array_equal(pl.count.cpu().numpy(), count)
    assert np.array_equal(pl.d.cpu().numpy(), d)
    tiles = ((W + 15) // 16) * ((H + 15) // 16)
    got_order, got, seg = api.lf_mpi_tile_lists(r.ws, n, tiles, N)
    assert np.array_equal(got_order, order)
    want, start = _lists(dict(order=order, chunk=chunk, rect=rect), W, H, N)
    seg = seg.astype(np.int64)
    ln = np.maximum(seg[:, 1] - seg[:, 0], 0)
    assert np.array_equal(ln, np.diff(start)) and len(got) == len(want)
    at = np.repeat(seg[:, 0] - start[:-1], ln) + np.arange(len(want))
    assert np.array_equal(got[at], want)


# sizes around one sort block (2048 and 4096 keys), around 152 blocks of four
# CTAs (one and four primitives per thread: 155,648) and around one wave of
# 4-key threads (311,296); a sort of one, two and three digits per tile key
# (up to 256, up to 65,536 and more super-tiles of 32 x 32), with and without
# more super-tiles than a block counts one by one (1024)
@pytest.mark.parametrize("n,size,N,binning,ties", [
    (1, (97, 33), 3, "quantile", 0),
    (2047, (512, 512), 5, "disparity", 0),
    (2049, (513, 512), 5, "quantile", 7),
    (4097, (1024, 1024), 128, "quantile", 100),
    (155648, (300, 200), 64, "disparity", 0),
    (155649, (300, 200), 64, "disparity", 5000),
    (155649, (1088, 1000), 33, "quantile", 3),
    (311297, (1024, 1024), 16, "quantile", 0),
    (40000, (8224, 8192), 1, "quantile", 0),
])
def test_order_planes_and_lists(orc, n, size, N, binning, ties):
    _check(orc, _scene(n, n + N, ties), orc.gauss_decide, size, N, binning, "u8" if size[0] > 8000 else "f16")


def test_disparity_bins_at_their_edges(orc):
    """Depths on and next to the edges of the disparity bins (one FP32 step
    either way), where an FP32 estimate of the bin alone would be wrong."""
    N, zn, zf = 64, 1.0, 9.0
    sc = _scene(20000, 5, 0)
    k = np.arange(20000)
    back = orc.make_ref(S.identity_camera(256), S.display_for(3.0, 0.1)).D_forward   # depths are taken from here
    ia, ib = 1.0 / (zn - back), 1.0 / (zf - back)
    edge = 1.0 / (ia - (k % (N + 1)) / N * (ia - ib)) + back
    z = edge.astype(np.float32)
    z = np.where(k % 3 == 0, z, np.nextafter(z, np.where(k % 3 == 1, np.float32(0), np.float32(99))))
    sc.means[:, :2] *= (z / sc.means[:, 2])[:, None]
    sc.means[:, 2] = np.clip(z, zn, zf)
    _check(orc, sc, orc.gauss_decide, (256, 256), N, "disparity")


@pytest.mark.parametrize("base,origin", [(1.0, (-0.4, -0.4, 1.5)), (0.3, (0.0, 0.0, 2.0)), (2.0 ** -1000, (0.1, 0.0, 2.0)),
                                         (1e30, (0.0, 0.0, 3.0))])
def test_voxel_projection_on_number_bits(orc, base, origin):
    """Levels from 0 to 255, indices of every size and sign, sides down to the
    subnormals: the projection's exponent and rounding steps give the FP64 and
    FP32 results bit for bit."""
    rng = np.random.default_rng(11)
    n = 6000
    level = rng.integers(0, 256, n) if base != 1.0 else rng.integers(0, 13, n)
    lim = np.minimum(2.0 ** np.minimum(level, 30), 2.0 ** 31 - 1)
    ijk = np.floor(rng.uniform(-1.0, 1.0, (n, 3)) * lim[:, None]).astype(np.int32)
    ijk[:40] = 0
    sc = S.VoxelScene(ijk, level.astype(np.uint8), np.asarray(origin, np.float64), float(base), np.ones((n, 8), np.float32),
                      np.full((n, 3), 0.5, np.float32))
    _check(orc, sc, orc.voxel_decide, (200, 150), 4, "quantile")
