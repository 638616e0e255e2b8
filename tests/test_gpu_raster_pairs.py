"""The paired Gaussian raster at its edges: list lengths around a staged batch and the parts that
long lists are cut into, planes that end inside a block of 8 x 8 pixels, and
colours that are not finite."""
import numpy as np
import pytest
import torch

from paper_2508_18540_gb300 import api
from paper_2508_18540_gb300 import synth as S
from tests import gpu_util as G

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2508_18540_gb300 import build
    build.build()


def _setup(size):
    cam = S.Camera(np.eye(3), np.zeros(3), np.radians(50.0), np.radians(50.0), *size)
    return cam, S.display_for(3.0, 0.05), S.ViewSet(1, 1)


def _scene(n, seed, scale):
    rng = np.random.default_rng(seed)
    z = rng.uniform(2.0, 5.0, n)
    xy = rng.uniform(-0.45, 0.45, (n, 2)) * z[:, None]
    f = np.float32
    return S.GaussianScene(np.column_stack([xy, z]).astype(f), np.exp(rng.normal(np.log(scale), 0.7, (n, 3))).astype(f),
                           rng.normal(size=(n, 4)).astype(f), rng.uniform(0.01, 0.3, n).astype(f),
                           rng.uniform(0.0, 1.0, (n, 3)).astype(f))


# FP32 planes against the FP64 oracle: max-abs 1e-4, as everywhere in these tests
@pytest.mark.parametrize("n", [1, 255, 256, 257, 512, 513, 1500])
@pytest.mark.parametrize("size", [(9, 17), (33, 31)])
def test_list_lengths_around_parts(orc, n, size):
    cam, disp, views = _setup(size)
    sc = _scene(n, n, 0.2)      # about a third of the plane each: nearly every list is n long
    o = orc.render(scene=sc, camera=cam, display=disp, views=views, N=1, binning="quantile")
    gpu = G.run_gpu(sc, cam, disp, views, 1, "quantile")
    assert gpu["status"] == 0 and np.array_equal(gpu["order"], o["order"])
    assert np.abs(gpu["planes"] - o["planes"]).max() <= 1e-4


@pytest.mark.parametrize("blend", ["exact", "3dgs"])
@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_colour_that_is_not_finite_stays_in_its_footprint(blend, bad):
    cam, disp, views = _setup((70, 50))
    sc = _scene(60, 9, 0.03)
    out = []
    for colour in (0.25, bad):
        sc.rgb[::7, 1] = colour
        r = api.LightFieldRenderer(cam, disp, views, 3, "quantile", "f32", blend=blend)
        pl = r.build(api.DeviceGaussians.from_scene(sc))
        assert r.status()[0] == 0
        out.append((pl.rgba.cpu().numpy(), pl.rect[:sc.n].cpu().numpy(), pl.chunk[:sc.n].cpu().numpy()))
    (a, rect, chunk), (b, _, _) = out
    inside = np.zeros(a.shape[:3], bool)
    for g in range(0, sc.n, 7):
        x0, y0, x1, y1 = rect[g]
        if chunk[g] >= 0:
            inside[chunk[g], y0:y1 + 1, x0:x1 + 1] = True
    assert inside.any() and not inside.all()
    same = a.view(np.int32) == b.view(np.int32)
    assert same[~inside].all()                       # outside: bit for bit
    assert same[..., [0, 2, 3]].all()                # the other channels everywhere
    changed = ~same[..., 1]
    assert changed.any() and not np.isfinite(b[..., 1][changed]).any()


@pytest.mark.parametrize("corner", [(-0.4, -0.4), (0.1, -0.4), (0.1, 0.1)])
def test_voxel_batches_without_hits(orc, corner):
    """All voxels of a super-tile lie in one of its four tiles: the other
    tiles go through several staged batches of its list without a hit."""
    rng = np.random.default_rng(3)
    n, cell = 1400, 0.04
    cam, disp, views = _setup((32, 32))
    ijk = np.floor(rng.uniform(0.0, 0.3, (n, 3)) / cell).astype(np.int32)
    sc = S.VoxelScene(ijk, np.zeros(n, np.uint8), np.array([2 * corner[0], 2 * corner[1], 2.0]), cell,
                      rng.uniform(0.0, 0.3, (n, 8)).astype(np.float32), rng.uniform(0.0, 1.0, (n, 3)).astype(np.float32))
    o = orc.render(scene=sc, camera=cam, display=disp, views=views, N=1, binning="quantile")
    gpu = G.run_gpu(sc, cam, disp, views, 1, "quantile")
    assert gpu["status"] == 0 and np.array_equal(gpu["rect"], o["rect"])
    assert np.abs(gpu["planes"] - o["planes"]).max() <= 1e-4   # FP32 planes, as above
