"""The build's waits for the sums of earlier blocks (depth sort, binning and
pair emission, sort of the pairs) when they give up: the call returns, the
host reads LF_ERR_TIMEOUT, the planes are empty, nothing is written out of
range, and the next build on the same workspace is right."""
import numpy as np
import pytest
import torch

from paper_2508_18540_gb300 import _lib as L
from paper_2508_18540_gb300 import api
from paper_2508_18540_gb300 import synth as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2508_18540_gb300 import build
    build.build()


def _scene(n, radius):
    rng = np.random.default_rng(n)
    z = rng.uniform(1.0, 9.0, n)
    xy = rng.uniform(-0.4, 0.4, (n, 2)) * z[:, None]
    f = np.float32
    return S.GaussianScene(np.column_stack([xy, z]).astype(f), (radius * z[:, None] * np.ones(3)).astype(f),
                           rng.normal(size=(n, 4)).astype(f), rng.uniform(0.1, 0.9, n).astype(f),
                           rng.uniform(0, 1, (n, 3)).astype(f))


# what waits first: the depth sort (more than 2048 keys), the binning (up to
# 2048 keys, more than 256 ranks), the pairs' sort (more than 2048 pairs of up
# to 256 ranks)
CASES = [("sort", 10000, 0.01, 200), ("sort", 200000, 0.003, 200), ("bin", 1500, 0.01, 200), ("tiles", 200, 0.1, 512)]


@pytest.mark.parametrize("first,n,radius,size", CASES)
@pytest.mark.parametrize("binning", ["quantile", "disparity"])
def test_build_waits_that_give_up(first, n, radius, size, binning):
    args = (S.identity_camera(size, 50.0), S.display_for(3.0, 0.1), S.ViewSet(3), 16, binning, "f32")
    g = api.DeviceGaussians.from_scene(_scene(n, radius))
    fresh = api.LightFieldRenderer(*args)
    want = fresh.build(g)
    st, pairs, M = fresh.status()
    assert st == L.LF_OK and M > 0.9 * n
    if first == "tiles":
        assert pairs > 2048
    r = api.LightFieldRenderer(*args)
    r._ensure(n)
    r.ws.fill_(0xff)   # what the lost entries' places hold
    for t in (r.planes.rgba, r.planes.d, r.planes.count):
        t.fill_(7)
    api.lf_selftest_build_waits(g, r.ref, r.N, binning, r.ws, r.planes)
    torch.cuda.synchronize()
    assert r.status()[0] == L.LF_ERR_TIMEOUT
    assert b"gave up" in L.load().lf_last_error()
    for t in (r.planes.rgba, r.planes.d, r.planes.count):
        assert not t.any()
    # the adjoint of the empty planes: no gradient, whatever the lost places hold
    # (the voxels' adjoint reads the same header and order)
    dplanes = torch.ones((r.N, r.ref.H, r.ref.W, 4), dtype=torch.float32, device="cuda")
    v = api.DeviceVoxels.from_scene(S.VoxelScene(np.zeros((n, 3), np.int32), np.zeros(n, np.uint8), np.zeros(3), 1.0,
                                                 np.ones((n, 8), np.float32), np.ones((n, 3), np.float32)))
    gg, gv = api.GaussianGrads.empty(n, "cuda"), api.VoxelGrads.empty(n, "cuda")
    fields = list(vars(gg).values()) + list(vars(gv).values())
    for t in fields:
        t.fill_(3)
    api.lf_build_mpi_backward_gaussians(g, r.ref, r.planes, dplanes, gg, r.ws)
    api.lf_build_mpi_backward_voxels(v, r.ref, r.planes, dplanes, gv, r.ws)
    torch.cuda.synchronize()
    for t in fields:
        assert not t.any()
    again = r.build(g)
    assert r.status() == (L.LF_OK, pairs, M)
    for a, b in zip((again.rgba, again.d, again.count, again.chunk, again.rect),
                    (want.rgba, want.d, want.count, want.chunk, want.rect)):
        assert torch.equal(a, b)


def test_batch_status_after_a_build_that_gave_up():
    wls = [S.workload_display(seed=30 + i, n=n, res=64, N=8, V=5) for i, n in enumerate((5000, 3000))]
    b = api.BatchRenderer(wls, "f32")
    b.render()
    assert b.status() == L.LF_OK
    want = [o.clone() for o in b.outputs]
    r, g, planes = b.parts[1]
    api.lf_selftest_build_waits(g, r.ref, r.N, wls[1].binning, r.ws, planes, b.stream)
    assert b.status() == L.LF_ERR_TIMEOUT
    b.render()
    assert b.status() == L.LF_OK
    for o, w in zip(b.outputs, want):
        assert torch.equal(o, w)
    b.close()
