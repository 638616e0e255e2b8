"""The one-walk plane filter against the two-pass one, which takes a plane that
is filtered alone: the same sums in the same order, so the same bits."""
import pytest
import torch

from paper_2508_18540_gb300 import api

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2508_18540_gb300 import build
    build.build()


def _planes(rgba, dtype):
    n = rgba.shape[0]
    d = torch.ones(n, dtype=torch.float64, device="cuda")
    count = torch.ones(n, dtype=torch.int32, device="cuda")
    members = torch.zeros(1, dtype=torch.int32, device="cuda"), torch.zeros(1, 4, dtype=torch.int32, device="cuda")
    return api.Planes(rgba, d, count, *members, api.DTYPES[dtype])


# widths around one strip of 64 columns and up to eight, heights around a band
# of 16 rows, radii on both sides of the two ring sizes (8, 9)
@pytest.mark.parametrize("dtype", ["f32", "f16", "bf16", "u8"])
@pytest.mark.parametrize("W,H,N,radius", [(1, 5, 310, 3), (63, 16, 304, 1), (65, 33, 160, 9), (130, 17, 110, 8),
                                          (448, 15, 45, 16), (511, 70, 40, 3), (512, 1, 40, 2), (512, 130, 38, 16)])
def test_one_walk_equals_two_passes(dtype, W, H, N, radius):
    gen = torch.Generator(device="cuda").manual_seed(W + H + radius)
    rgba = torch.rand(N, H, W, 4, device="cuda", generator=gen)
    rgba = (255 * rgba).to(torch.uint8) if dtype == "u8" else rgba.to(api.TORCH_DTYPES[api.DTYPES[dtype]])
    if dtype != "u8":
        rgba[0, H // 2, W // 2, 1] = float("inf")
    apart = rgba.clone()
    api.lf_filter_planes(_planes(rgba, dtype), radius / 3.0, radius)
    for k in range(N):
        api.lf_filter_planes(_planes(apart[k:k + 1], dtype), radius / 3.0, radius)
    assert torch.equal(rgba.view(torch.uint8), apart.view(torch.uint8))
