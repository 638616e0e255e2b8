"""Timed work of the framework: light-field frames, plane building, compositing and fitting steps.

A case is a dict of plain values; `kind` says which public call it is:

  frame      one light-field frame of Gaussians or voxels (LightFieldRenderer.render, or replay of its captured graph)
  splat      the sweeping planes alone (LightFieldRenderer.build)
  composite  the quilt views of planes that are in hand (LightFieldRenderer.composite's call, api.lf_composite)
  fit        a frame and its gradients (LightFieldRenderer.render and .backward)
  batch      several scenes as one frame (BatchRenderer.launch of its captured graph)

Inputs are drawn on the GPU from the seed: Gaussians in blobs or in a box, sparse voxels of a smooth noise field, and for
the composite planes of soft textured blobs.
"""
from __future__ import annotations

import math

import torch
import torch.nn.functional as F

from paper_2508_18540_gb300 import api
from paper_2508_18540_gb300 import synth as S

DEV = "cuda"


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def _case(kind, **kw):
    """A case with every field that its kind reads."""
    c = {"kind": kind, "prims": "blobs", "n": 100_000, "Nx": 512, "Ny": 512, "P_s": 1, "N": 64, "binning": "quantile",
         "Vx": 45, "Vy": 1, "atlas": 0, "bilinear": False, "dtype": "f32", "blend": "exact", "filter": 0.0,
         "replay": False, "save": True}
    c.update(kw)
    return c


def listed():
    """Twelve calls over the range of sizes, types and directions."""
    return [
        # the smallest configuration: a preview frame, launches and latency count
        _case("frame", name="frame_tiny", prims="box", n=10_000, Nx=128, Ny=128, N=16, Vx=9, binning="disparity"),
        # the display-scale frame as a render loop runs it: one captured graph replayed
        _case("frame", name="frame_display_1m", n=1_000_000, replay=True),
        # a 48-view two-dimensional quilt of odd size, FP16 planes, written as one atlas image
        _case("frame", name="frame_quilt_f16_odd", n=60_000, Nx=427, Ny=241, N=48, Vx=8, Vy=6, atlas=8, dtype="f16"),
        # plane building at twice the view resolution with many planes, 16-bit planes
        _case("splat", name="splat_ps2_n128_bf16", n=500_000, P_s=2, N=128, dtype="bf16"),
        # plane building with the 3DGS rasteriser's cut-offs
        _case("splat", name="splat_3dgs_300k", n=300_000, blend="3dgs"),
        # sparse voxels at display scale with the low-pass filter that replaces supersampling
        _case("frame", name="frame_voxels_2m_filter", prims="voxels", n=2_000_000, filter=0.7),
        # compositing alone (a static scene seen on a display that changes), FP32 planes, nearest
        _case("composite", name="composite_f32"),
        # the smoother sampling option, FP16 planes
        _case("composite", name="composite_bilinear_f16", bilinear=True, dtype="f16"),
        # the largest plane set, RGBA8 planes (the compact format), twice the view resolution and 90 views
        _case("composite", name="composite_u8_ps2_n256", P_s=2, N=256, Vx=90, dtype="u8"),
        # one fitting step of 300k Gaussians with the saved composite state
        _case("fit", name="fit_gaussians_300k", n=300_000),
        # one fitting step of voxels, bilinear sampling, no saved state, few small views
        _case("fit", name="fit_voxels_bilinear", prims="voxels", n=100_000, Nx=256, Ny=256, N=32, Vx=9, bilinear=True,
              save=False),
        # three uneven scenes as one batched frame, FP16 planes
        _case("batch", name="batch_uneven_f16", n="50000,200000,500000", Nx="256,384,512", Ny="256,384,512",
              N="64,64,128", Vx="9,45,45", dtype="f16"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _cost(c):
    """Rough work of a case: (pixel, member) pairs and (pixel, plane) view samples, more of them where a gradient is
    asked for or a plane row is not a multiple of 16 bytes."""
    total = 0.0
    times = {"fit": 8.0 if c["save"] else 14.0, "batch": 2.0}.get(c["kind"], 1.0)
    for q in _scenes(c):
        W, H = q["Nx"] * q["P_s"], q["Ny"] * q["P_s"]
        pairs = 0.0 if q["kind"] == "composite" else q["n"] * 235.0 * (W * H / 512.0 ** 2)
        samples = 0.0 if q["kind"] == "splat" else float(q["Nx"] * q["Ny"] * q["Vx"] * q["Vy"]) * q["N"]
        ragged = W * {"f32": 16, "u8": 4}.get(q["dtype"], 8) % 16 != 0
        samples *= (2.0 if q["bilinear"] else 1.0) * (4.0 if ragged else 1.0)
        total += times * (2.0 * pairs + samples) + 2.0 * q["N"] * W * H
    return total


def draw(rng):
    """One more case of the listed ranges."""
    most = max(_cost(c) for c in listed())
    while True:
        kind = rng.choice(["frame", "frame", "frame", "splat", "splat", "composite", "composite", "composite", "fit",
                           "fit", "batch"])
        side = lambda: _log_int(rng, 96, 768)  # noqa: E731
        Nx = side()
        Ny = Nx if rng.random() < 0.4 else min(768, max(96, int(Nx * rng.uniform(0.5, 1.6))))
        Vx, Vy = rng.choice([(rng.randint(1, 96), 1), (rng.randint(2, 11), rng.randint(2, 8))])
        c = _case(kind, n=_log_int(rng, 5_000, 1_500_000), Nx=Nx, Ny=Ny, N=_log_int(rng, 8, 256), Vx=Vx, Vy=Vy,
                  P_s=rng.choice([1, 1, 1, 2]), bilinear=rng.random() < 0.35,
                  binning=rng.choice(["quantile", "quantile", "disparity"]))
        if kind == "frame":
            c["prims"] = rng.choice(["blobs", "blobs", "box", "voxels"])
            c["dtype"] = rng.choice(["f32", "f16"])
            c["replay"] = rng.random() < 0.5
            c["atlas"] = Vx if rng.random() < 0.3 else 0
            c["filter"] = rng.choice([0.0, 0.5, 0.7, 1.2]) if c["prims"] == "voxels" else 0.0
            c["blend"] = "3dgs" if c["prims"] != "voxels" and c["dtype"] == "f32" and rng.random() < 0.2 else "exact"
        elif kind == "splat":
            c["prims"] = rng.choice(["blobs", "blobs", "box", "voxels"])
            c["dtype"] = rng.choice(["f32", "f16", "bf16"])
            c["blend"] = "3dgs" if c["prims"] != "voxels" and rng.random() < 0.3 else "exact"
        elif kind == "composite":
            c["dtype"] = rng.choice(["f32", "f16", "bf16", "u8"])
            c["atlas"] = Vx if rng.random() < 0.2 else 0
        elif kind == "fit":
            c["prims"] = rng.choice(["blobs", "blobs", "voxels"])
            c["n"] = _log_int(rng, 5_000, 400_000)
            c["save"] = rng.random() < 0.7
        else:
            k = rng.randint(2, 4)
            several = lambda f: ",".join(str(f()) for _ in range(k))  # noqa: E731
            c.update(n=several(lambda: _log_int(rng, 5_000, 500_000)), N=several(lambda: _log_int(rng, 8, 128)),
                     Vx=several(lambda: rng.randint(1, 60)), Nx=several(lambda: 8 * _log_int(rng, 12, 80)), Vy=1, P_s=1,
                     dtype=rng.choice(["f32", "f16"]))
            c["Ny"] = several(lambda: _log_int(rng, 96, 640))
        if _cost(c) <= 0.9 * most:
            return c


def _scenes(c):
    """The scenes of a case: one, or a batch's, each with numbers in place of the lists."""
    if c["kind"] != "batch":
        return [c]
    cols = {k: [int(v) for v in str(c[k]).split(",")] for k in ("n", "Nx", "Ny", "N", "Vx")}
    return [dict(c, kind="frame", **{k: v[i] for k, v in cols.items()}) for i in range(len(cols["n"]))]


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _setup(c):
    """Camera, display and view set of one scene: 50 degrees, a +-0.15 baseline (+-0.06 up and down with several view
    rows), the focal distance at the disparity centre of the scene's depths."""
    th = math.radians(50.0)
    thy = 2.0 * math.atan(math.tan(th / 2) * c["Ny"] / c["Nx"])
    voxels = c["prims"] == "voxels"
    z0, z1 = _depths(c)
    cam = S.Camera(torch.eye(3, dtype=torch.float64).numpy(), torch.tensor([0.0, 0.0, 6.0 if voxels else 0.0],
                   dtype=torch.float64).numpy(), th, thy, c["Nx"], c["Ny"])
    focal = 2.0 / (1.0 / z0 + 1.0 / z1)
    base = 0.1 if c["prims"] == "box" else 0.15
    disp = S.Display(D_focal=focal, phi_x=2.0 * math.atan(base / focal),
                     phi_y=2.0 * math.atan(0.06 / focal) if c["Vy"] > 1 else 0.0, P_s=c["P_s"])
    return cam, disp, S.ViewSet(c["Vx"], c["Vy"], c["bilinear"], (0.0, 0.0, 0.0), c["atlas"])


def _depths(c):
    return {"voxels": (4.0, 8.0), "box": (2.0, 6.0)}.get(c["prims"], (1.5, 10.0))


def _rand(gen, *shape):
    return torch.rand(*shape, generator=gen, device=DEV)


def _gaussians(c, gen):
    """Blobs: 200 clusters over depth 1.5 .. 10, anisotropic, Beta(2, 2) opacities. Box: isotropic, uniform in a box."""
    n = c["n"]
    rn = lambda *s: torch.randn(*s, generator=gen, device=DEV)  # noqa: E731
    if c["prims"] == "box":
        means = torch.cat([2.0 * _rand(gen, n, 2) - 1.0, 2.0 + 4.0 * _rand(gen, n, 1)], 1)
        scales = torch.exp(math.log(0.02) + 0.3 * rn(n, 1)).expand(n, 3)
        quats = torch.tensor([1.0, 0.0, 0.0, 0.0], device=DEV).expand(n, 4)
        op = 0.1 + 0.8 * _rand(gen, n)
    else:
        tx = math.tan(math.radians(25.0))
        ty = tx * c["Ny"] / c["Nx"]
        cz = 1.5 + 8.5 * _rand(gen, 200)
        cx, cy = ((1.6 * _rand(gen, 200) - 0.8) * cz * t for t in (tx, ty))
        blob = torch.arange(n, device=DEV) % 200
        means = torch.stack([cx, cy, cz], 1)[blob] + rn(n, 3) * (0.05 * cz[blob])[:, None]
        scales = torch.exp(math.log(0.01) + 0.5 * rn(n, 3))
        quats = F.normalize(rn(n, 4), dim=1)
        op = torch.sort(_rand(gen, n, 3), dim=1).values[:, 1].clamp(1e-3, 0.999)   # the middle of three: Beta(2, 2)
    return api.DeviceGaussians(*(t.float().contiguous() for t in (means, scales, quats, op, _rand(gen, n, 3))))


def _voxels(c, gen):
    """The cells of a 256^3 grid over [-2, 2]^3 where a smooth noise field is highest, the highest of them split into 8
    (one cell in twelve); softplus(N(0, 2)) corner densities."""
    n, res = c["n"], 256 if c["n"] > 150_000 else 96
    field = 0.0
    for r, amp in ((8, 1.0), (24, 0.5), (64, 0.25)):
        lat = amp * torch.randn(1, 1, r + 1, r + 1, r + 1, generator=gen, device=DEV)
        field = field + F.interpolate(lat, size=(res, res, res), mode="trilinear", align_corners=True)
    split = n // 12
    keep = n - 7 * split
    order = torch.topk(field.reshape(-1), keep).indices
    cell = lambda i: torch.stack([i // (res * res), (i // res) % res, i % res], 1)  # noqa: E731
    child = torch.tensor([[i & 1, (i >> 1) & 1, (i >> 2) & 1] for i in range(8)], device=DEV)
    fine = (2 * cell(torch.sort(order[:split]).values)[:, None, :] + child).reshape(-1, 3)
    coarse = cell(torch.sort(order[split:]).values)
    ijk = torch.cat([coarse, fine]).int()
    level = torch.cat([torch.zeros(coarse.shape[0], device=DEV), torch.ones(fine.shape[0], device=DEV)]).to(torch.uint8)
    m = ijk.shape[0]
    dens = F.softplus(2.0 * torch.randn(m, 8, generator=gen, device=DEV))
    return api.DeviceVoxels(ijk.contiguous(), level, dens.contiguous(), _rand(gen, m, 3), (-2.0, -2.0, -2.0), 4.0 / res)


def _prims(c, gen):
    return _voxels(c, gen) if c["prims"] == "voxels" else _gaussians(c, gen)


def _planes(c, gen):
    """Planes in hand (texels, distances, member counts): each a dozen soft blobs with a textured opacity, about one
    plane in sixteen empty, at unevenly spaced depths."""
    N, H, W = c["N"], c["Ny"] * c["P_s"], c["Nx"] * c["P_s"]
    z0, z1 = _depths(c)
    u = torch.sort(_rand(gen, N).double()).values
    d = z0 + (z1 - z0) * (0.15 * u + 0.85 * (torch.arange(N, device=DEV) + 0.5) / N)
    count = (_rand(gen, N) > 1.0 / 16).int() * 1000
    count[0] = 1000
    rgba = torch.zeros(N, H, W, 4, dtype=api.TORCH_DTYPES[api.DTYPES[c["dtype"]]], device=DEV)
    ys, xs = (torch.arange(m, device=DEV, dtype=torch.float32) / m for m in (H, W))
    for k, full in enumerate(count.tolist()):
        if not full:
            continue
        b = _rand(gen, 5, 12)
        sd = 0.03 + 0.04 * b[2]
        ey = torch.exp(-0.5 * ((ys[:, None] - (0.05 + 0.9 * b[0])) / sd) ** 2) * (0.5 + 3.0 * b[3])
        ex = torch.exp(-0.5 * ((xs[:, None] - (0.05 + 0.9 * b[1])) / sd) ** 2)
        tex = F.interpolate(_rand(gen, 1, 4, max(2, H // 6), max(2, W // 6)), size=(H, W), mode="bilinear",
                            align_corners=True)[0]
        a = 1.0 - torch.exp(-(ey @ ex.T) * (0.3 + 1.4 * tex[3]))
        a = torch.where(a < 1.0 / 512, torch.zeros_like(a), a)
        t = torch.stack([a * tex[0], a * tex[1], a * tex[2], a], -1)
        rgba[k] = torch.round(255.0 * t).to(torch.uint8) if c["dtype"] == "u8" else t.to(rgba.dtype)
    return rgba, d, count


class _Scene:
    """A scene description in host memory, as BatchRenderer takes it."""

    def __init__(self, c, gen):
        self.camera, self.display, self.views = _setup(c)
        self.N, self.binning = c["N"], c["binning"]
        g = _gaussians(c, gen)
        self.scene = S.GaussianScene(*(t.cpu().numpy() for t in (g.means, g.scales, g.quats, g.opacity, g.rgb)))


def prepare(case, seed):
    """The primitives or planes, and the renderer with its buffers (and captured graph) that a program keeps."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed))
    c = case
    if c["kind"] == "batch":
        batch = api.BatchRenderer([_Scene(q, gen) for q in _scenes(c)], c["dtype"])
        batch.capture()
        batch.synchronize()
        return {"case": c, "batch": batch}
    cam, disp, views = _setup(c)
    s = {"case": c, "views": views}
    if c["kind"] == "composite":
        s["ref"] = api.lf_make_ref_camera(cam, disp)
        rgba, d, count = _planes(c, gen)
        members = torch.zeros(1, dtype=torch.int32, device=DEV), torch.zeros(1, 4, dtype=torch.int32, device=DEV)
        s["planes"] = api.Planes(rgba, d, count, *members, api.DTYPES[c["dtype"]])
        s["ws"] = api.alloc_workspace(api.lf_composite_workspace_size(c["N"], views))
        s["out"] = torch.empty(api.views_shape(views, c["Nx"], c["Ny"]), dtype=torch.float32, device=DEV)
        return s
    s["prims"] = _prims(c, gen)
    s["r"] = api.LightFieldRenderer(cam, disp, views, c["N"], c["binning"], c["dtype"], n_capacity=s["prims"].n,
                                    plane_filter=c["filter"], blend=c["blend"],
                                    save_state=c["kind"] == "fit" and c["save"])
    if c["kind"] == "fit":
        s["dviews"] = 0.05 * torch.randn(c["Vx"] * c["Vy"], c["Ny"], c["Nx"], 4, generator=gen, device=DEV)
    if c["replay"] and c["kind"] == "frame":
        s["r"].capture(s["prims"])
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(state):
    c = state["case"]
    if c["kind"] == "batch":
        b = state["batch"]
        b.launch()
        torch.cuda.current_stream().wait_stream(b.stream)
        return b.outputs
    if c["kind"] == "composite":
        api.lf_composite(state["planes"], state["ref"], state["views"], state["out"], state["ws"])
        return state["out"]
    r, prims = state["r"], state["prims"]
    if c["kind"] == "splat":
        pl = r.build(prims)
        return {"rgba": pl.rgba, "d": pl.d, "count": pl.count, "chunk": pl.chunk, "rect": pl.rect}
    views = r.replay() if c["replay"] and c["kind"] == "frame" else r.render(prims)
    if c["kind"] == "frame":
        return views
    grads, dplanes = r.backward(prims, state["dviews"])
    return {"views": views, "dplanes": dplanes, "grads": list(vars(grads).values())}


# ---------------------------------------------------------------------------
# the work that a pass cannot do without
# ---------------------------------------------------------------------------

def _pairs(c):
    """(pixel, primitive) pairs of the footprints, estimated from a sample of the scene."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(1)
    ref = _Ref(c)
    m = min(c["n"], 20_000)
    if c["prims"] == "voxels":
        v = _voxels(c, gen)
        rect, ok = _decide_voxels(ref, v)[1:3]
    else:
        rect, ok = _decide_gaussians(ref, _gaussians(dict(c, n=m), gen))[1:3]
    r = rect.double()
    area = (r[:, 2] - r[:, 0] + 1) * (r[:, 3] - r[:, 1] + 1) * ok
    return float(area.mean()) * c["n"]


def work(case):
    """Inputs and outputs moved once; 15 operations a (pixel, Gaussian) pair, 95 a (pixel, voxel) pair, 8 a nearest and
    20 a bilinear (view pixel, plane) sample; a backward pass three times its forward; 4 (2 r + 1) a filtered texel
    and axis."""
    nbytes = flops = 0.0
    for c in _scenes(case):
        tb = {"f32": 16, "u8": 4}.get(c["dtype"], 8)
        texels = float(c["N"] * c["Nx"] * c["Ny"] * c["P_s"] ** 2)
        views = float(c["Vx"] * c["Vy"] * c["Nx"] * c["Ny"])
        prim = 57.0 if c["prims"] == "voxels" else 56.0
        sweep = views * c["N"] * (20.0 if c["bilinear"] else 8.0)
        if c["kind"] == "composite":
            nbytes += texels * tb + 16 * views
            flops += sweep
            continue
        splat = _pairs(c) * (95.0 if c["prims"] == "voxels" else 15.0)
        if c["filter"]:
            splat += texels * 4 * 2 * 2 * (2 * math.ceil(3 * c["filter"]) + 1)
        nbytes += prim * c["n"]
        flops += splat
        if c["kind"] == "splat":
            nbytes += texels * tb + 20 * c["n"]
            continue
        nbytes += 16 * views
        flops += sweep
        if c["kind"] == "fit":
            nbytes += 16 * views + 16 * texels + prim * c["n"]
            flops += 3 * (sweep + splat)
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# ---------------------------------------------------------------------------
# Whole-number decisions (footprints, chunks, nearest texels) are taken in the precision that the interface prescribes
# for them (include/lf.h); every value is computed in 64 bits.

def _fma(a, b, c):
    """a b + c in FP32, rounded once (the product is exact in FP64)."""
    d = lambda v: v.double() if torch.is_tensor(v) else float(v)  # noqa: E731
    return (d(a) * d(b) + d(c)).float()


def _f32(v):
    return float(torch.tensor(v, dtype=torch.float64).float())


class _Ref:
    """The reference camera of one scene: moved forward along +z so that every view's frustum is covered."""

    def __init__(self, c):
        cam, disp, self.views = _setup(c)
        self.c, self.Nx, self.Ny, self.P_s, self.N = c, c["Nx"], c["Ny"], c["P_s"], c["N"]
        self.W, self.H = self.Nx * self.P_s, self.Ny * self.P_s
        self.Df = disp.D_focal
        self.tth = [math.tan(0.5 * cam.theta_x), math.tan(0.5 * cam.theta_y)]
        self.tphi = [math.tan(0.5 * disp.phi_x), math.tan(0.5 * disp.phi_y)]
        self.fwd = max(self.Df * p / (p + t) if p > 0 else 0.0 for p, t in zip(self.tphi, self.tth))
        self.tthp = [self.Df * t / (self.Df - self.fwd) for t in self.tth]
        self.f = [self.W / (2 * self.tthp[0]), self.H / (2 * self.tthp[1])]
        self.ctr = [0.5 * (self.W - 1), 0.5 * (self.H - 1)]
        ratio = self.Df * self.tth[0] / ((self.Df - self.fwd) * self.tthp[0]) * self.P_s
        self.fp = disp.f_aa * ratio * ratio
        self.t2 = float(cam.t[2])
        self.near = disp.z_near


def _clip_rect(ref, fx0, fy0, fx1, fy1):
    ok = (fx0 <= ref.W - 1) & (fx1 >= 0) & (fy0 <= ref.H - 1) & (fy1 >= 0)
    rect = torch.stack([fx0.clamp(min=0), fy0.clamp(min=0), fx1.clamp(max=ref.W - 1), fy1.clamp(max=ref.H - 1)], 1)
    return rect, ok


def _rotation(q):
    w, x, y, z = q.unbind(1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3)


def _decide_gaussians(ref, g):
    """Reference depth (FP64), clipped footprint and culling of every Gaussian; the footprint in FP32, in the order of
    operations that fixes its bits (the camera axes are the world's)."""
    z = (g.means[:, 2].double() + ref.t2) - ref.fwd
    xc, yc, zc = g.means[:, 0], g.means[:, 1], z.float()
    q = g.quats
    n2 = _fma(q[:, 0], q[:, 0], _fma(q[:, 1], q[:, 1], _fma(q[:, 2], q[:, 2], q[:, 3] * q[:, 3])))
    q = q * (torch.ones_like(n2) / torch.sqrt(n2))[:, None]
    V = _rotation(q) * g.scales[:, None, :]
    iz = torch.ones_like(zc) / zc
    xn, yn = xc * iz, yc * iz
    fx, fy = (_f32(v) for v in ref.f)
    U0 = (fx * iz)[:, None] * _fma(-xn[:, None], V[:, 2], V[:, 0])
    U1 = (fy * iz)[:, None] * _fma(-yn[:, None], V[:, 2], V[:, 1])

    def dot(a, b):
        return _fma(a[:, 0], b[:, 0], _fma(a[:, 1], b[:, 1], a[:, 2] * b[:, 2]))

    fp = _f32(ref.fp)
    s00, s01, s11 = dot(U0, U0) + fp, dot(U0, U1), dot(U1, U1) + fp
    det = _fma(s00, s11, -(s01 * s01))
    mid = 0.5 * (s00 + s11)
    lam = mid + torch.sqrt(_fma(mid, mid, -det).clamp(min=0))
    rad = torch.ceil(3.0 * torch.sqrt(lam))
    px, py = _fma(fx, xn, _f32(ref.ctr[0])), _fma(fy, yn, _f32(ref.ctr[1]))
    rect, ok = _clip_rect(ref, torch.ceil(px - rad), torch.ceil(py - rad), torch.floor(px + rad), torch.floor(py + rad))
    return z, rect, ok & (det > 0) & (z > ref.near)


def _voxel_boxes(v):
    side = v.base_size * torch.pow(2.0, -v.level.double())
    return torch.tensor(v.origin, device=DEV, dtype=torch.float64) + v.ijk.double() * side[:, None], side


def _decide_voxels(ref, v):
    lo, side = _voxel_boxes(v)
    z = (lo[:, 2] + 0.5 * side + ref.t2) - ref.fwd
    ok = z - 0.5 * side > ref.near
    fx, fy = (_f32(f) for f in ref.f)
    px, py = [], []
    for k in range(8):
        X, Y, Z = ((lo[:, a] + ((k >> a) & 1) * side).float() for a in range(3))
        iz = torch.ones_like(Z) / (Z + _f32(ref.t2 - ref.fwd))
        px.append(_fma(fx, X * iz, _f32(ref.ctr[0])))
        py.append(_fma(fy, Y * iz, _f32(ref.ctr[1])))
    px, py = torch.stack(px), torch.stack(py)
    x0, x1 = torch.ceil(px.amin(0)), torch.floor(px.amax(0))
    y0, y1 = torch.ceil(py.amin(0)), torch.floor(py.amax(0))
    rect, inside = _clip_rect(ref, x0, y0, x1, y1)
    return z, rect, ok & inside & (x0 <= x1) & (y0 <= y1)


def _bins(ref, z, ok):
    """Depth order, first rank of every chunk, member counts and plane distances."""
    idx = torch.nonzero(ok).squeeze(1)
    idx = idx[torch.sort(z[idx], stable=True).indices]
    zs, M, N = z[idx], idx.numel(), ref.N
    if M == 0:
        return idx, [0] * (N + 1), torch.zeros(N, dtype=torch.float64, device=DEV)
    if ref.c["binning"] == "quantile":
        chunk = torch.arange(M, device=DEV) * N // M
    else:
        i0, i1 = 1.0 / zs[0], 1.0 / zs[-1]
        chunk = torch.floor(N * (i0 - 1.0 / zs) / (i0 - i1)).clamp(max=N - 1).long()
    start = torch.searchsorted(chunk, torch.arange(N + 1, device=DEV)).tolist()
    if ref.c["binning"] == "quantile":
        d = [0.0 if a == b else float(0.5 * (zs[(a + b - 1) // 2] + zs[(a + b) // 2])) + ref.fwd
             for a, b in zip(start, start[1:])]
        d = torch.tensor(d, dtype=torch.float64, device=DEV)
    else:
        d = 1.0 / (i0 - (torch.arange(N, device=DEV).double() + 0.5) / N * (i0 - i1)) + ref.fwd
    return idx, start, d


def _members(rect, W):
    """Every (member, pixel) pair of one chunk, grouped by pixel and in depth order within a pixel."""
    x0, y0, x1, y1 = rect.long().unbind(1)
    w = x1 - x0 + 1
    area = w * (y1 - y0 + 1)
    m = torch.repeat_interleave(torch.arange(area.numel(), device=DEV), area)
    j = torch.arange(m.numel(), device=DEV) - torch.repeat_interleave(torch.cumsum(area, 0) - area, area)
    x, y = x0[m] + j % w[m], y0[m] + j // w[m]
    p = y * W + x
    p, order = torch.sort(p, stable=True)
    return m[order], x[order], y[order], p


def _blend(ref, p, neglog, colour, H, W, cut=False):
    """Front to back "over" of pairs grouped by pixel p: neglog = -log(1 - alpha), colour per pair. [H, W, 4]."""
    out = torch.zeros(H * W, 4, dtype=torch.float64, device=DEV)
    if p.numel() == 0:
        return out.view(H, W, 4)
    first = torch.ones_like(p, dtype=torch.bool)
    first[1:] = p[1:] != p[:-1]
    seg = torch.cumsum(first, 0) - 1
    incl = torch.cumsum(neglog, 0)
    start = (incl - neglog)[first][seg]
    behind = incl - start
    if cut:
        keep = torch.exp(-behind) >= 1e-4
        neglog = torch.where(keep, neglog, torch.zeros_like(neglog))
    alpha = -torch.expm1(-neglog)
    T = torch.exp(-(behind - neglog))
    rgb = (T * alpha)[:, None] * colour
    out = out.index_add(0, p, torch.cat([rgb, neglog[:, None]], 1))
    return torch.cat([out[:, :3], -torch.expm1(-out[:, 3:])], 1).view(H, W, 4)


def _project(ref, g):
    """2D mean and conic of the EWA projection (FP64): g = (means, scales, quats) as FP64 tensors."""
    means, scales, quats = g
    x, y, z = means[:, 0], means[:, 1], means[:, 2] + ref.t2 - ref.fwd
    V = _rotation(quats / quats.norm(dim=1, keepdim=True)) * scales[:, None, :]
    U0 = (ref.f[0] / z)[:, None] * (V[:, 0] - (x / z)[:, None] * V[:, 2])
    U1 = (ref.f[1] / z)[:, None] * (V[:, 1] - (y / z)[:, None] * V[:, 2])
    s00, s01, s11 = (U0 * U0).sum(1) + ref.fp, (U0 * U1).sum(1), (U1 * U1).sum(1) + ref.fp
    det = s00 * s11 - s01 * s01
    mean = torch.stack([ref.f[0] * x / z + ref.ctr[0], ref.f[1] * y / z + ref.ctr[1]], 1)
    return mean, torch.stack([s11 / det, -s01 / det, s00 / det], 1)


def _gauss_plane(ref, rect, mean, conic, op, rgb):
    m, x, y, p = _members(rect, ref.W)
    dx, dy = x - mean[m, 0], y - mean[m, 1]
    q = conic[m, 0] * dx * dx + 2 * conic[m, 1] * dx * dy + conic[m, 2] * dy * dy
    a = (op[m] * torch.exp(-0.5 * q)).clamp(max=0.99)
    cut = ref.c["blend"] == "3dgs"
    if cut:
        a = torch.where(a < 1.0 / 255, torch.zeros_like(a), a)
    return _blend(ref, p, -torch.log1p(-a), rgb[m], ref.H, ref.W, cut)


def _voxel_plane(ref, rect, lo, side, dens, rgb):
    m, x, y, p = _members(rect, ref.W)
    d = torch.stack([(x - ref.ctr[0]) / ref.f[0], (y - ref.ctr[1]) / ref.f[1], torch.ones_like(x).double()], 1)
    d = d / d.norm(dim=1, keepdim=True)
    o = torch.tensor([0.0, 0.0, ref.fwd - ref.t2], dtype=torch.float64, device=DEV)
    b, s = lo[m] - o, side[m]
    ta, tb = b / d, (b + s[:, None]) / d
    t0 = torch.minimum(ta, tb).nan_to_num(nan=-math.inf).amax(1).clamp(min=0)
    t1 = torch.maximum(ta, tb).nan_to_num(nan=math.inf).amin(1)
    hit = (t1 > t0) & torch.isfinite(t1)
    length = torch.where(hit, t1 - t0, torch.zeros_like(t0))
    t0 = torch.where(hit, t0, torch.zeros_like(t0))

    def density(t):
        f = ((t[:, None] * d - b) / s[:, None]).clamp(0, 1)
        g = 1 - f
        acc = 0.0
        for k in range(8):
            wk = 1.0
            for a in range(3):
                wk = wk * (f[:, a] if (k >> a) & 1 else g[:, a])
            acc = acc + wk * dens[m, k]
        return acc

    integral = length / 6 * (density(t0) + 4 * density(t0 + 0.5 * length) + density(t0 + length))
    return _blend(ref, p, integral, rgb[m], ref.H, ref.W)


def _filter64(planes, sigma):
    r = math.ceil(3 * sigma)
    t = torch.arange(-r, r + 1, dtype=torch.float64, device=DEV)
    w = torch.exp(-0.5 * (t / sigma) ** 2)
    w = w / w.sum()
    for k in range(planes.shape[0]):
        x = planes[k].permute(2, 0, 1)[:, None]
        x = F.conv2d(F.conv2d(x, w.view(1, 1, 1, -1), padding=(0, r)), w.view(1, 1, -1, 1), padding=(r, 0))
        planes[k] = x[:, 0].permute(1, 2, 0)
    return planes


class _Splat64:
    """The planes of a scene in 64 bits, and the gradients of its parameters from those of the planes."""

    def __init__(self, ref, prims):
        self.ref, self.prims = ref, prims
        self.voxels = ref.c["prims"] == "voxels"
        z, rect, ok = (_decide_voxels if self.voxels else _decide_gaussians)(ref, prims)
        self.idx, self.start, self.d = _bins(ref, z, ok)
        self.rect = rect[self.idx]
        if self.voxels:
            lo, side = _voxel_boxes(prims)
            self.fixed = (lo[self.idx], side[self.idx])
            self.leaves = [prims.density8.double(), prims.rgb.double()]
        else:
            self.leaves = [t.double() for t in (prims.means, prims.scales, prims.quats, prims.opacity, prims.rgb)]

    def values(self):
        """Per member, in depth order: the tensors that the planes are functions of."""
        if self.voxels:
            return [t[self.idx] for t in self.leaves]
        means, scales, quats, op, rgb = (t[self.idx] for t in self.leaves)
        mean, conic = _project(self.ref, (means, scales, quats))
        return [mean, conic, op, rgb]

    def plane(self, k, vals):
        a, b = self.start[k], self.start[k + 1]
        part = [v[a:b] for v in vals]
        if self.voxels:
            return _voxel_plane(self.ref, self.rect[a:b], *(v[a:b] for v in self.fixed), *part)
        return _gauss_plane(self.ref, self.rect[a:b], *part)

    def planes(self):
        vals = self.values()
        return torch.stack([self.plane(k, vals) for k in range(self.ref.N)])

    def count(self):
        return [b - a for a, b in zip(self.start, self.start[1:])]

    def grads(self, dplanes):
        self.leaves = [t.requires_grad_(True) for t in self.leaves]
        vals = self.values()
        mid = [v.detach().requires_grad_(True) for v in vals]
        for k in range(self.ref.N):
            if self.start[k + 1] > self.start[k]:
                self.plane(k, mid).backward(dplanes[k])
        torch.autograd.backward(vals, [torch.zeros_like(v) if v.grad is None else v.grad for v in mid])
        return [t.grad for t in self.leaves]


def _axis(ref, axis, j, V, d, n, Wp):
    """gm, hn of the FP32 nearest decision and the FP64 sample positions along one axis for views j, planes d."""
    s = 0.0 if V <= 1 else j / (V - 1) - 0.5
    delta = 2.0 * ref.Df * s * ref.tphi[axis]
    den = (d - ref.fwd) * ref.tthp[axis]
    a = d * ref.tth[axis]
    g = Wp * a / (n * den)
    hn = 0.5 * Wp * ((delta * (ref.Df - d) / ref.Df + a * (1 - n) / n) / den + 1.0)
    return (g - ref.P_s).float(), hn.float(), g, hn - 0.5


class _Sampler:
    """Samples of one view: plane texels at nearest or bilinear positions, zero outside; and the adjoint of that."""

    def __init__(self, ref, d, v):
        self.ref = ref
        vs = ref.views
        i, j = v // vs.Vx, v % vs.Vx
        self.x = self.taps(_axis(ref, 0, j, vs.Vx, d, ref.Nx, ref.W), ref.Nx, ref.W)
        self.y = self.taps(_axis(ref, 1, i, vs.Vy, d, ref.Ny, ref.H), ref.Ny, ref.H)

    def taps(self, coef, n, size):
        """[(index, weight)] per tap, each [N, n]; weight 0 outside the plane."""
        gm, hn, g, hb = (t[:, None] for t in coef)
        x = torch.arange(n, device=DEV)
        if not self.ref.views.bilinear:
            idx = [self.ref.P_s * x + torch.floor(_fma(gm, x.float(), hn)).long()]
            wt = [torch.ones_like(idx[0], dtype=torch.float64)]
        else:
            X = g * x + hb
            lo = torch.floor(X)
            idx, wt = [lo.long(), lo.long() + 1], [1.0 - (X - lo), X - lo]
        inside = [(q >= 0) & (q < size) for q in idx]
        return [(q.clamp(0, size - 1), w * ok) for q, w, ok in zip(idx, wt, inside)]

    def __call__(self, plane, k):
        out = 0.0
        for iy, wy in self.y:
            rows = plane[iy[k]]
            for ix, wx in self.x:
                out = out + (wy[k][:, None] * wx[k])[..., None] * rows[:, ix[k]]
        return out

    def scatter(self, dplane, k, grad):
        flat = dplane.view(-1, 4)
        for iy, wy in self.y:
            for ix, wx in self.x:
                flat.index_add_(0, (iy[k][:, None] * self.ref.W + ix[k]).reshape(-1),
                                ((wy[k][:, None] * wx[k])[..., None] * grad).reshape(-1, 4))


def _atlas(ref, views):
    """Views [V, Ny, Nx, 4] as the quilt image, where the case asks for one."""
    c = ref.views.atlas_cols
    if not c:
        return views
    V, Ny, Nx = views.shape[:3]
    rows = (V + c - 1) // c
    return views.view(rows, c, Ny, Nx, 4).permute(0, 2, 1, 3, 4).reshape(rows * Ny, c * Nx, 4)


def _composite64(ref, planes, d, count, dviews=None):
    """Views of the planes; with dviews, also the gradient of the planes."""
    live = [k for k in range(ref.N) if count[k]]
    V = ref.views.Vx * ref.views.Vy
    out = torch.zeros(V, ref.Ny, ref.Nx, 4, dtype=torch.float64, device=DEV)
    dplanes = None if dviews is None else torch.zeros_like(planes)
    for v in range(V):
        s = _Sampler(ref, d, v)
        T = torch.ones(ref.Ny, ref.Nx, dtype=torch.float64, device=DEV)
        kept = []
        for k in live:
            t = s(planes[k].double(), k)
            out[v, ..., :3] += T[..., None] * t[..., :3]
            if dviews is not None:
                kept.append((t, T))
            T = T * (1.0 - t[..., 3])
        out[v, ..., 3] = 1.0 - T
        if dviews is not None:
            g = dviews[v].double()
            B = -g[..., 3]
            for k, (t, Tk) in zip(reversed(live), reversed(kept)):
                s.scatter(dplanes[k], k, torch.cat([Tk[..., None] * g[..., :3], (-Tk * B)[..., None]], -1))
                B = (t[..., :3] * g[..., :3]).sum(-1) + (1.0 - t[..., 3]) * B
    return _atlas(ref, out), dplanes


def exact(case, seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed))
    c = case
    if c["kind"] == "composite":
        ref = _Ref(c)
        rgba, d, count = _planes(c, gen)
        rgba = rgba.double().div_(255.0) if c["dtype"] == "u8" else rgba
        return _composite64(ref, rgba, d, count.tolist())[0]
    got = []
    for q in _scenes(c):
        ref = _Ref(q)
        sp = _Splat64(ref, _prims(q, gen))
        planes = sp.planes()
        if c["kind"] == "splat":
            return {"rgba": planes, "d": sp.d, "count": None, "chunk": None, "rect": None}
        if q["filter"]:
            planes = _filter64(planes, q["filter"])
        if c["kind"] == "fit":
            dv = 0.05 * torch.randn(c["Vx"] * c["Vy"], c["Ny"], c["Nx"], 4, generator=gen, device=DEV)
            views, dplanes = _composite64(ref, planes, sp.d, sp.count(), dv)
            return {"views": views, "dplanes": dplanes, "grads": sp.grads(dplanes)}
        got.append(_composite64(ref, planes, sp.d, sp.count())[0])
    return got if c["kind"] == "batch" else got[0]
