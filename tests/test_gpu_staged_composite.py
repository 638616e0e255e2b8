"""The staged composite and its adjoint at the edges of their layout, on planes
that are in hand: plane rows that are not multiples of 16 bytes, tiles of 128,
64 and 32 columns, windows wider than a stage (planes close to the reference
camera), more planes than descriptors, views that end early, empty planes.

Views against the FP64 oracle's composite of the same texels: nearest within
1e-4 (the decisions are the same, the sums FP32); bilinear within 1e-3: a
sample position is FP32 and below 4096 here, so its weights are within 2^-12,
and at most 7 planes of texels within [0, 0.3] add up. dplanes against FP64
autograd of the same sampling: 2e-5 and 1e-3 of the largest gradient.
"""
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
    assert torch.cuda.is_available(), "GPU tests need CUDA"


@pytest.fixture(scope="module")
def orc():
    import oracle
    return oracle


def _case(dtype, P_s, Nx, Ny, views, N, opaque_from=None, seed=0):
    cam = S.Camera(np.eye(3), np.zeros(3), np.radians(50.0), np.radians(40.0), Nx, Ny)
    disp = S.display_for(3.0, 0.15, P_s=P_s, phi_y=0.02)
    ref = api.lf_make_ref_camera(cam, disp)
    rng = np.random.default_rng(seed)
    t = rng.uniform(0.0, 0.3, (N, ref.H, ref.W, 4)).astype(np.float32)
    if opaque_from is not None:
        t[opaque_from:, :, :, 3] = 1.0
    # from close to the reference camera (wide windows) to far behind the focus
    d = ref.D_forward + np.geomspace(0.15, 20.0, N)
    count = np.ones(N, np.int32)
    count[1::5] = 0
    if dtype == "u8":
        rgba = torch.from_numpy(np.round(t * 255).astype(np.uint8)).cuda()
        vals = rgba.double().cpu().numpy() / 255
    else:
        rgba = torch.from_numpy(t).cuda().to(api.TORCH_DTYPES[api.DTYPES[dtype]])
        vals = rgba.double().cpu().numpy()
    pl = api.Planes(rgba, torch.from_numpy(d).cuda(), torch.from_numpy(count).cuda(),
                    torch.zeros(1, dtype=torch.int32, device="cuda"),
                    torch.zeros((1, 4), dtype=torch.int32, device="cuda"), api.DTYPES[dtype])
    ws = api.alloc_workspace(api.lf_composite_workspace_size(N, views))
    return cam, disp, ref, pl, vals, d, count, ws


SHAPES = [("f32", 1, 128, 5, 45, 1), ("f16", 1, 67, 9, 8, 2), ("u8", 1, 33, 6, 16, 1), ("bf16", 2, 131, 4, 10, 3),
          ("f32", 3, 160, 3, 2, 1), ("u8", 1, 515, 2, 1, 1), ("f16", 1, 20, 11, 5, 1), ("f32", 1, 300, 2, 3, 1)]


@pytest.mark.parametrize("bilinear", [False, True])
@pytest.mark.parametrize("dtype,P_s,Nx,Ny,Vx,Vy", SHAPES)
def test_views_against_oracle(orc, dtype, P_s, Nx, Ny, Vx, Vy, bilinear):
    views = S.ViewSet(Vx, Vy, bilinear, (0.1, 0.2, 0.3))
    cam, disp, ref, pl, vals, d, count, ws = _case(dtype, P_s, Nx, Ny, views, 7)
    out = torch.full(api.views_shape(views, Nx, Ny), float("nan"), device="cuda")
    api.lf_composite(pl, ref, views, out, ws)
    assert api.lf_composite_status(7, views, ws) == 0
    want = orc.composite(orc.make_ref(cam, disp), vals, d, count, Vx, Vy, bilinear, views.bg)
    assert float(np.abs(out.cpu().numpy() - want).max()) <= (1e-3 if bilinear else 1e-4)
    # the saving form blends the same texels
    state = torch.empty(api.composite_state_shape(ref, views), device="cuda")
    api.lf_composite_save(pl, ref, views, out, state, ws)
    assert float(np.abs(out.cpu().numpy() - want).max()) <= (1e-3 if bilinear else 1e-4)


@pytest.mark.parametrize("dtype,Nx,opaque_from", [("f32", 200, 9), ("u8", 131, 3), ("f16", 64, 66), ("bf16", 33, 40)])
def test_views_that_end_early(orc, dtype, Nx, opaque_from):
    # 70 planes, opaque from one on: every view stops there and the tiles end
    views = S.ViewSet(17, 1)
    cam, disp, ref, pl, vals, d, count, ws = _case(dtype, 1, Nx, 6, views, 70, opaque_from, seed=3)
    out = torch.full(api.views_shape(views, Nx, 6), float("nan"), device="cuda")
    api.lf_composite(pl, ref, views, out, ws)
    assert api.lf_composite_status(70, views, ws) == 0
    want = orc.composite(orc.make_ref(cam, disp), vals, d, count, 17, 1, False, views.bg)
    assert float(np.abs(out.cpu().numpy() - want).max()) <= 1e-4


def _adjoint64(orc, cam, disp, vals, d, count, views, dviews):
    """dplanes of the plain composite by FP64 autograd, sampled where the oracle says."""
    ref = orc.make_ref(cam, disp)
    N, H, W = vals.shape[:3]
    planes = torch.from_numpy(vals).requires_grad_(True)
    dx, dy = orc.view_offsets(ref, views.Vx, views.Vy)

    def taps(axis, delta, dk, n, size):
        if not views.bilinear:
            gm, hn, _ = orc.axis_coeffs(ref, axis, delta, dk)
            i0 = torch.tensor([orc.nearest_index(ref, gm, hn, x) for x in range(n)])
            pairs = [(i0, torch.ones(n, dtype=torch.float64))]
        else:
            X = torch.tensor([orc.plane_pixel(ref, axis, delta, dk, x) for x in range(n)], dtype=torch.float64)
            lo = torch.floor(X)
            pairs = [(lo.long(), 1 - (X - lo)), (lo.long() + 1, X - lo)]
        return [(i.clamp(0, size - 1), w * ((i >= 0) & (i < size))) for i, w in pairs]

    loss = 0.0
    for v in range(views.Vx * views.Vy):
        i, j = divmod(v, views.Vx)
        Q, T = torch.zeros(cam.Ny, cam.Nx, 3, dtype=torch.float64), torch.ones(cam.Ny, cam.Nx, dtype=torch.float64)
        for k in range(N):
            if not count[k]:
                continue
            t = 0.0
            for iy, wy in taps(1, dy[i], d[k], cam.Ny, H):
                for ix, wx in taps(0, dx[j], d[k], cam.Nx, W):
                    t = t + (wy[:, None] * wx)[..., None] * planes[k][iy][:, ix]
            Q = Q + T[..., None] * t[..., :3]
            T = T * (1 - t[..., 3])
        g = dviews[v].double().cpu()
        out = torch.cat([Q + T[..., None] * torch.tensor(views.bg, dtype=torch.float64), (1 - T)[..., None]], -1)
        loss = loss + (g * out).sum()
    loss.backward()
    return planes.grad.numpy()


@pytest.mark.parametrize("bilinear", [False, True])
@pytest.mark.parametrize("dtype,P_s,Nx,Ny,Vx,Vy", [("f32", 1, 130, 3, 10, 1), ("f16", 1, 67, 5, 4, 2),
                                                   ("u8", 2, 33, 4, 9, 1), ("f32", 3, 160, 2, 2, 1)])
def test_adjoint_against_autograd(orc, dtype, P_s, Nx, Ny, Vx, Vy, bilinear):
    views = S.ViewSet(Vx, Vy, bilinear, (0.1, 0.2, 0.3))
    cam, disp, ref, pl, vals, d, count, ws = _case(dtype, P_s, Nx, Ny, views, 7, seed=5)
    gen = torch.Generator(device="cuda").manual_seed(3)
    dv = torch.randn((Vx * Vy, Ny, Nx, 4), device="cuda", generator=gen)
    want = _adjoint64(orc, cam, disp, vals, d, count, views, dv)
    got = torch.full(vals.shape, float("nan"), device="cuda")
    api.lf_composite_backward(pl, ref, views, dv, got, ws)
    tol = (1e-3 if bilinear else 2e-5) * np.abs(want).max()
    assert np.abs(got.cpu().numpy() - want).max() <= tol
    out = torch.empty(api.views_shape(views, Nx, Ny), device="cuda")
    state = torch.empty(api.composite_state_shape(ref, views), device="cuda")
    api.lf_composite_save(pl, ref, views, out, state, ws)
    got.fill_(float("nan"))
    api.lf_composite_backward_saved(pl, ref, views, dv, state, got, ws)
    assert api.lf_composite_status(7, views, ws) == 0
    assert np.abs(got.cpu().numpy() - want).max() <= tol
