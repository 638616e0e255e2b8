"""The composite adjoint where its walks end early: opaque texels, more planes
than descriptors in shared memory, views past one group, ragged rows. References
and tolerances are those of test_gpu_staged_composite (FP64 autograd)."""
import numpy as np
import pytest
import torch

from paper_2508_18540_gb300 import api
from paper_2508_18540_gb300 import synth as S
from tests.test_gpu_staged_composite import _adjoint64, _built, _case, orc  # noqa: F401

pytestmark = pytest.mark.gpu


# On rows of whole 16-byte words the adjoint leaves the colours behind an opaque
# texel out of its alpha gradient where no pixel of the warp goes further: there
# the alpha gradients of opaque texels are not compared.
# opaque: the share of opaque 4 x 4 blocks in every plane, or the plane from
# which on every texel is opaque; planes in all (90: of these 72 not empty)
@pytest.mark.parametrize("bilinear", [False, True])
@pytest.mark.parametrize("dtype,Nx,Vx,N,opaque", [
    ("f32", 64, 4, 12, 0.5), ("f16", 64, 4, 12, 0.9), ("f16", 67, 4, 12, 0.5), ("u8", 67, 4, 12, 0.9),
    ("f32", 40, 12, 90, 0.02), ("bf16", 41, 12, 90, 0.02), ("f32", 130, 5, 14, 3), ("u8", 33, 11, 90, 70)])
def test_opaque_texels_against_autograd(orc, dtype, Nx, Vx, N, opaque, bilinear):  # noqa: F811
    views = S.ViewSet(Vx, 1, bilinear, (0.1, 0.2, 0.3))
    Ny = 4
    cam, disp, ref, pl, vals, d, count, ws = _case(dtype, 1, Nx, Ny, views, N, seed=5)
    rng = np.random.default_rng(1)
    if isinstance(opaque, float):
        hit = rng.random((N, (Ny + 3) // 4, (Nx + 3) // 4)) < opaque
        hit = np.repeat(np.repeat(hit, 4, 1), 4, 2)[:, :Ny, :Nx]
    else:
        hit = np.zeros(vals.shape[:3], bool)
        hit[opaque:] = True
    pl.rgba[..., 3][torch.from_numpy(hit).cuda()] = 255 if dtype == "u8" else 1.0
    vals[..., 3][hit] = 1.0
    gen = torch.Generator(device="cuda").manual_seed(3)
    dv = torch.randn((Vx, Ny, Nx, 4), device="cuda", generator=gen)
    want = _adjoint64(orc, cam, disp, vals, d, count, views, dv)
    tol = (1e-3 if bilinear else 2e-5) * np.abs(want).max()
    whole_words = Nx * pl.rgba.element_size() * 4 % 16 == 0

    def error():
        e = np.abs(got.cpu().numpy() - want)
        if whole_words:
            assert np.isfinite(e).all()
            e[..., 3][hit] = 0.0
        return e.max()

    got = torch.full(vals.shape, float("nan"), device="cuda")
    api.lf_composite_backward(pl, ref, views, dv, got, ws)
    assert api.lf_composite_status(N, views, ws) == 0
    assert error() <= tol
    out = torch.empty(api.views_shape(views, Nx, Ny), device="cuda")
    state = torch.empty(api.composite_state_shape(ref, views), device="cuda")
    api.lf_composite_save(pl, ref, views, out, state, ws)
    got.fill_(float("nan"))
    api.lf_composite_backward_saved(pl, ref, views, dv, state, got, ws)
    assert api.lf_composite_status(N, views, ws) == 0
    assert error() <= tol


@pytest.mark.parametrize("saved", [False, True])
@pytest.mark.parametrize("dtype,Nx", [("f16", 67), ("bf16", 41), ("u8", 33)])
def test_transmittance_on_ragged_rows_is_divided(orc, dtype, Nx, saved):  # noqa: F811
    """T in front of every plane, read off dL/dC of one pixel in every sixth row
    (they share no texel) with g = 1, against the same walks with FP32 divisions: within 2 ulp. (Each step may
    miss the rounded quotient by little more than half an ulp; reciprocals
    without a correction drift by 5 ulp and more over 50 planes.)"""
    views, N, Ny, x0 = S.ViewSet(1, 1), 62, 48, Nx // 2
    cam, disp, ref, pl, vals, d, count, ws = _case(dtype, 1, Nx, Ny, views, N, seed=9)
    dv = torch.zeros((1, Ny, Nx, 4), device="cuda")
    dv[0, ::6, x0, 0] = 1.0
    got = torch.empty(vals.shape, device="cuda")
    if saved:
        out = torch.empty(api.views_shape(views, Nx, Ny), device="cuda")
        state = torch.empty(api.composite_state_shape(ref, views), device="cuda")
        api.lf_composite_save(pl, ref, views, out, state, ws)
        api.lf_composite_backward_saved(pl, ref, views, dv, state, got, ws)
    else:
        api.lf_composite_backward(pl, ref, views, dv, got, ws)
    got = got.cpu().numpy()
    o = orc.make_ref(cam, disp)
    dx, dy = orc.view_offsets(o, 1, 1)
    f, checked = np.float32, 0
    A = vals[..., 3].astype(f)
    if dtype == "u8":   # decoded by a product
        A = np.round(255 * vals[..., 3]).astype(f) * f(1.0 / 255.0)
    for y in range(0, Ny, 6):
        walk = []   # (plane, row, column, 1 - A) in order
        for k in np.flatnonzero(count):
            gx, hx, _ = orc.axis_coeffs(o, 0, dx[0], d[k])
            gy, hy, _ = orc.axis_coeffs(o, 1, dy[0], d[k])
            ix, iy = orc.nearest_index(o, gx, hx, x0), orc.nearest_index(o, gy, hy, y)
            if 0 <= ix < Nx and 0 <= iy < vals.shape[1]:
                walk.append((k, iy, ix, f(1) - A[k, iy, ix]))
        T = f(1)
        for _, _, _, a in walk:
            T = f(T * a)
        if saved:   # the saving forward's T behind the last plane
            T = f(state[0, y, x0, 0].item())
        for k, iy, ix, a in reversed(walk):
            T = f(T / a)
            assert abs(got[k, iy, ix, 0] - T) <= 2.0 ** -22 * T, (y, k)
            checked += 1
    assert checked > 40 * Ny // 6
