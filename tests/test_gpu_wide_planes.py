"""Composite and adjoint of planes many times as wide as the view, whose windows
are cut to the shared memory that there is. References and tolerances are those
of test_gpu_staged_composite."""
import numpy as np
import pytest
import torch

from paper_2508_18540_gb300 import api
from paper_2508_18540_gb300 import synth as S
from tests.test_gpu_staged_composite import _adjoint64, _built, _case, orc  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bilinear", [False, True])
@pytest.mark.parametrize("dtype,P_s,Nx,Vx", [("f32", 8, 256, 9), ("f32", 8, 256, 3), ("f32", 16, 250, 9), ("f32", 10, 200, 45),
                                             ("f16", 16, 255, 15), ("u8", 16, 129, 1), ("f32", 16, 256, 2)])
def test_views_against_oracle(orc, dtype, P_s, Nx, Vx, bilinear):  # noqa: F811
    views = S.ViewSet(Vx, 1, bilinear, (0.1, 0.2, 0.3))
    cam, disp, ref, pl, vals, d, count, ws = _case(dtype, P_s, Nx, 2, views, 7)
    want = orc.composite(orc.make_ref(cam, disp), vals, d, count, Vx, 1, bilinear, views.bg)
    out = torch.full(api.views_shape(views, Nx, 2), float("nan"), device="cuda")
    api.lf_composite(pl, ref, views, out, ws)
    assert api.lf_composite_status(7, views, ws) == 0
    assert float(np.abs(out.cpu().numpy() - want).max()) <= (1e-3 if bilinear else 1e-4)
    state = torch.empty(api.composite_state_shape(ref, views), device="cuda")
    api.lf_composite_save(pl, ref, views, out, state, ws)
    assert float(np.abs(out.cpu().numpy() - want).max()) <= (1e-3 if bilinear else 1e-4)


@pytest.mark.parametrize("bilinear", [False, True])
@pytest.mark.parametrize("P_s,Nx,Vx", [(8, 130, 9), (16, 130, 3)])
def test_adjoint_against_autograd(orc, P_s, Nx, Vx, bilinear):  # noqa: F811
    views = S.ViewSet(Vx, 1, bilinear, (0.1, 0.2, 0.3))
    cam, disp, ref, pl, vals, d, count, ws = _case("f32", P_s, Nx, 1, views, 6, seed=5)
    gen = torch.Generator(device="cuda").manual_seed(3)
    dv = torch.randn((Vx, 1, Nx, 4), device="cuda", generator=gen)
    want = _adjoint64(orc, cam, disp, vals, d, count, views, dv)
    got = torch.full(vals.shape, float("nan"), device="cuda")
    api.lf_composite_backward(pl, ref, views, dv, got, ws)
    assert api.lf_composite_status(6, views, ws) == 0
    assert np.abs(got.cpu().numpy() - want).max() <= (1e-3 if bilinear else 2e-5) * np.abs(want).max()
