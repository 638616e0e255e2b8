"""3DGS blending on lists that go on long after their pixels have stopped, on
planes that end inside a block: texels away from the cut-offs' thresholds (the
oracle marks the others) within 1e-4 of the FP64 oracle, as in test_gpu_parity."""
import numpy as np
import pytest

from paper_2508_18540_gb300 import api
from tests.test_gpu_raster_pairs import _built, _scene, _setup  # noqa: F401

pytestmark = pytest.mark.gpu


# list lengths around the batches of 256 entries; opacities at which all pixels
# of a block stop in the first batch, in a later one, or in some blocks only
@pytest.mark.parametrize("n,opacity", [(256, 0.9), (257, 0.9), (700, 0.9), (2000, 0.05), (2000, 0.9)])
@pytest.mark.parametrize("size", [(9, 17), (64, 48), (70, 50)])
def test_long_lists_of_stopped_pixels(orc, n, opacity, size):
    cam, disp, views = _setup(size)
    sc = _scene(n, n, 0.2)
    sc.opacity[:] = opacity * (0.5 + sc.opacity)
    o = orc.render(scene=sc, camera=cam, display=disp, views=views, N=1, binning="quantile", with_views=False, blend="3dgs")
    r = api.LightFieldRenderer(cam, disp, views, 1, "quantile", "f32", blend="3dgs")
    pl = r.build(api.DeviceGaussians.from_scene(sc))
    assert r.status()[0] == 0
    far = ~o["near"].astype(bool)
    assert far.mean() > 0.2
    e = np.abs(pl.rgba.cpu().numpy().astype(np.float64) - o["planes"]).max(axis=-1)
    assert e[far.reshape(e.shape)].max() <= 1e-4
