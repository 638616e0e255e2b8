"""Launches of one kernel from several threads at once, each with a shared-memory
size of its own: none is refused."""
import ctypes
import threading

import pytest
import torch

from paper_2508_18540_gb300 import api
from paper_2508_18540_gb300 import synth as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2508_18540_gb300 import build
    build.build()


def _statuses(calls, times):
    """Runs every call `times` times, each in a thread of its own; the statuses seen."""
    seen = set()

    def work(call):
        try:
            seen.update(call() for _ in range(times))
        except Exception as e:  # noqa: BLE001
            seen.add(repr(e))

    threads = [threading.Thread(target=work, args=(c,)) for c in calls]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    return seen


# (a limit set to each launch's own size refused 3 % of the wider filters)
def test_plane_filters_of_different_radii():
    lib, keep, calls = api.load(), [], []
    for i in range(6):
        rgba = torch.rand(64, 4, 64, 4, device="cuda")
        planes = api.Planes(rgba, torch.ones(64, dtype=torch.float64, device="cuda"),
                            torch.ones(64, dtype=torch.int32, device="cuda"),
                            torch.zeros(1, dtype=torch.int32, device="cuda"),
                            torch.zeros(1, 4, dtype=torch.int32, device="cuda"), api.DTYPES["f32"])
        ps, stream, radius = planes.c_struct(), torch.cuda.Stream(), (1, 16)[i % 2]
        keep.append((planes, ps, stream))
        calls.append(lambda ps=ps, stream=stream, radius=radius: lib.lf_filter_planes(
            ctypes.byref(ps), radius / 3.0, radius, ctypes.c_void_p(stream.cuda_stream)))
    torch.cuda.synchronize()
    assert _statuses(calls, 5000) == {0}


def test_composites_of_different_windows():
    """The same kernels with windows of one and of eight plane texels per pixel."""
    parts = []
    for P_s, res in ((1, 48), (8, 48)) * 2:
        r = api.LightFieldRenderer(S.identity_camera(res, 50.0), S.display_for(3.0, 0.1, P_s=P_s),
                                   S.ViewSet(3, bilinear=True), 4, "quantile", "f32", save_state=True)
        r.build(api.DeviceGaussians.from_scene(S.workload_tiny().scene))
        parts.append((r, r.composite().clone(), torch.cuda.Stream()))
    torch.cuda.synchronize()
    assert _statuses([lambda r=r, s=s: r.composite(s) is r.out for r, _, s in parts], 1000) == {True}
    for r, want, _ in parts:
        assert torch.equal(r.out, want)
