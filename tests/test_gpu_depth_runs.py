"""The depth order of long runs of depths that the sort's 24-bit keys do not
tell apart, against the FP64 oracle (integers and FP64 bits: no tolerance)."""
import numpy as np
import pytest

from paper_2508_18540_gb300 import api
from paper_2508_18540_gb300 import synth as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2508_18540_gb300 import build
    build.build()


# runs sorted in shared memory (up to 2048 keys) and in global memory
@pytest.mark.parametrize("n", [33, 2048, 2049, 100000])
@pytest.mark.parametrize("order", ["shuffled", "last two swapped", "in order"])
def test_one_long_run_of_near_equal_depths(orc, n, order):
    """A camera turned by 1e-9 rad about y gives depth = z - 1e-9 x, so the n
    Gaussians at z = 4 are one run; two more span the depths."""
    th, N, f = 1e-9, 8, np.float32
    rng = np.random.default_rng(n)
    perm = rng.permutation(n) if order == "shuffled" else np.arange(n)
    if order == "last two swapped":
        perm[-2:] = perm[:-3:-1]
    m = np.column_stack([np.linspace(0.5, -0.5, n)[perm], rng.uniform(-0.3, 0.3, n), np.full(n, 4.0)])
    m = np.concatenate([m, [[0, 0, 1.2], [0, 0, 8]]]).astype(f)
    sc = S.GaussianScene(m, np.full((n + 2, 3), 0.002, f), rng.normal(size=(n + 2, 4)).astype(f),
                         np.full(n + 2, 0.5, f), np.full((n + 2, 3), 0.5, f))
    R = np.array([[np.cos(th), 0.0, np.sin(th)], [0.0, 1.0, 0.0], [-np.sin(th), 0.0, np.cos(th)]])
    cam = S.Camera(R, np.zeros(3), np.radians(50.0), np.radians(50.0), 96, 96)
    disp = S.display_for(3.0, 0.1)
    ref = orc.make_ref(cam, disp)
    z, valid, _ = orc.gauss_decide(ref, sc)
    want, chunk, d, count, M = orc.bin_primitives(ref, z, valid, N, "quantile")
    assert M == n + 2
    r = api.LightFieldRenderer(cam, disp, S.ViewSet(1, 1), N, "quantile", "f16")
    pl = r.build(api.DeviceGaussians.from_scene(sc))
    st, _, gm = r.status()
    assert st == 0 and gm == M
    got, _, _ = api.lf_mpi_tile_lists(r.ws, sc.n, 36, N)
    assert np.array_equal(got, want)
    assert np.array_equal(pl.chunk.cpu().numpy(), chunk)
    assert np.array_equal(pl.count.cpu().numpy(), count)
    assert np.array_equal(pl.d.cpu().numpy(), d)
