"""Bilinear composite and adjoint of few views that lie far apart, whose windows
are cut to what leaves room for the CTAs of an SM, on planes from close to the
reference camera (no window) to far away. References and tolerances are those of
test_gpu_staged_composite."""
import numpy as np
import pytest
import torch

from paper_2508_18540_gb300 import api
from paper_2508_18540_gb300 import synth as S
from tests.test_gpu_staged_composite import _adjoint64, _built, _case, orc  # noqa: F401

pytestmark = pytest.mark.gpu

# windows of all three widths: from 0.25, 0.35 and 0.5 of the focal distance on
SHAPES = [("f32", 1, 256, 5, 1), ("f32", 1, 256, 2, 1), ("f16", 1, 512, 3, 1), ("f32", 1, 323, 3, 2), ("u8", 1, 400, 2, 2),
          ("bf16", 1, 771, 5, 1), ("f32", 2, 260, 3, 1)]


@pytest.mark.parametrize("dtype,P_s,Nx,Vx,Vy", SHAPES)
def test_views_against_oracle(orc, dtype, P_s, Nx, Vx, Vy):  # noqa: F811
    views = S.ViewSet(Vx, Vy, True, (0.1, 0.2, 0.3))
    cam, disp, ref, pl, vals, d, count, ws = _case(dtype, P_s, Nx, 3, views, 7)
    want = orc.composite(orc.make_ref(cam, disp), vals, d, count, Vx, Vy, True, views.bg)
    out = torch.full(api.views_shape(views, Nx, 3), float("nan"), device="cuda")
    api.lf_composite(pl, ref, views, out, ws)
    assert api.lf_composite_status(7, views, ws) == 0
    assert float(np.abs(out.cpu().numpy() - want).max()) <= 1e-3
    state = torch.empty(api.composite_state_shape(ref, views), device="cuda")
    api.lf_composite_save(pl, ref, views, out, state, ws)
    assert float(np.abs(out.cpu().numpy() - want).max()) <= 1e-3


@pytest.mark.parametrize("dtype,P_s,Nx,Vx,Vy", [("f32", 1, 323, 3, 2), ("f16", 1, 131, 6, 1), ("f32", 2, 130, 3, 1)])
def test_adjoint_against_autograd(orc, dtype, P_s, Nx, Vx, Vy):  # noqa: F811
    views = S.ViewSet(Vx, Vy, True, (0.1, 0.2, 0.3))
    cam, disp, ref, pl, vals, d, count, ws = _case(dtype, P_s, Nx, 2, views, 7, seed=5)
    gen = torch.Generator(device="cuda").manual_seed(3)
    dv = torch.randn((Vx * Vy, 2, Nx, 4), device="cuda", generator=gen)
    want = _adjoint64(orc, cam, disp, vals, d, count, views, dv)
    got = torch.full(vals.shape, float("nan"), device="cuda")
    api.lf_composite_backward(pl, ref, views, dv, got, ws)
    assert api.lf_composite_status(7, views, ws) == 0
    assert np.abs(got.cpu().numpy() - want).max() <= 1e-3 * np.abs(want).max()
