"""The work that users of this package have it do, as measurable cases.

Each case is a dict of plain values; `prepare` builds what a program holds
before the call (inputs on the GPU, plans, workspaces), `run` makes one pass
through the public entry points, `work` says what a pass cannot do without and
`exact` gives the same outputs in 64 bits from plain torch, without this
package's code.  `draw` gives further cases of the same ranges.

Geometry: the volume spans about 400 x 400 x 200 mm (the small case 256 mm
cubed), seen by a circular cone-beam scan with SAD / SDD 1000 / 1500 mm on a
detector of about 397 x 298 mm, marched at half a voxel.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2503_22139_gb300 as pmf
from paper_2503_22139_gb300 import autograd as pag
from paper_2503_22139_gb300 import ops, pipeline

DT = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}
KAPPA = 3.0
SAD, SDD, SCAN = 1000.0, 1500.0, 660
STDS = (5.0, 2.0, 1.0)  # MBC vectors per level, mm


# ------------------------------------------------------------------ the cases

def listed():
    paper = dict(nx=200, ny=200, nz=100, voxel=2.0)
    det = dict(nu=512, nv=384, pitch=0.776, step=1.0)
    small = dict(nx=64, ny=64, nz=64, voxel=4.0, nu=128, nv=128, pitch=1.6, step=2.0)
    return [
        # one optimisation iteration of the paper-scale reconstruction (Stages 2-3): the native plan, replayed
        # from a graph, 32 projections, grids stored in bf16; the largest case
        dict(name="plan_paper_bf16_b32", kind="plan", **paper, **det, gauss=100000, m0=500, m1=2000, m2=8000,
             batch=32, dtype="bf16"),
        # the same model under torch.autograd on the small volume: what a user who trains their own encoder calls;
        # launches and host work count
        dict(name="autograd_small_f32", kind="autograd", **small, gauss=2000, m0=200, m1=0, m2=0, batch=8,
             dtype="f32"),
        # the reference volume of a reconstruction: 100,000 small Gaussians into bf16
        dict(name="voxelize_ref_100k_bf16", kind="vox", **paper, gauss=100000, channels=1, dtype="bf16"),
        # gradients of a motion level's 2,000 wide 3-vector Gaussians
        dict(name="voxelize_grad_mbc_2k", kind="voxgrad", **paper, gauss=2000, channels=3),
        # the warped volumes of a batch of 32, as the training step makes them (bf16 grids, fp32 volumes)
        dict(name="warp_bf16_b32", kind="warp", **paper, batch=32, dtype="bf16", out="f32"),
        # the warp's adjoint for a Stage-3 batch of 8, fp32 grids
        dict(name="warp_grad_f32_b8", kind="warpgrad", **paper, batch=8, dtype="f32"),
        # projections of 32 fp32 warped volumes
        dict(name="project_f32_b32", kind="proj", **paper, **det, batch=32, dtype="f32"),
        # their adjoint for a batch of 8
        dict(name="backproject_b8", kind="projgrad", **paper, **det, batch=8),
        # four patients' volumes of different, odd sizes in one launch each way (an odd x size has no 16-byte rows)
        dict(name="uneven_ragged_f32", kind="uneven", nx=203, ny=161, nz=87, voxel=2.0, nu=509, nv=379, pitch=0.776,
             step=1.0, items=4, batch=7, dtype="f32"),
        # the loss terms of Eq. 14 (L1, D-SSIM, TV crop, MBC normality) of a Stage-3 batch
        dict(name="eq14_terms_b8", kind="eq14", **paper, nu=512, nv=384, batch=8, crop=32, dtype="bf16"),
        # Stage 1: one rasterized view per iteration, replayed from a graph
        dict(name="stage1_b1", kind="stage1", **paper, **det, gauss=100000, batch=1, crop=32),
        # the unfused calls, one projection at a time: DVF, warp and both adjoints
        dict(name="unfused_f32_b1", kind="unfused", **paper, batch=1, dtype="f32"),
    ]


def _logi(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_grid(rng, lo, hi):
    nx = _logi(rng, lo, hi)
    ny = max(8, nx + rng.randint(-9, 9))
    nz = max(8, nx // 2 + rng.randint(-5, 5))
    return dict(nx=nx, ny=ny, nz=nz, voxel=round(400.0 / nx, 3))


def _draw_det(rng, voxel, lo=96, hi=512):
    nu = _logi(rng, lo, hi)
    nv = max(16, int(0.75 * nu) + rng.randint(-9, 9))
    return dict(nu=nu, nv=nv, pitch=round(397.0 / nu, 4), step=round(0.5 * voxel, 4))


def draw(rng):
    kind = rng.choice(["plan", "autograd", "vox", "voxgrad", "warp", "warpgrad", "proj", "projgrad", "uneven", "eq14",
                       "stage1", "unfused"])
    dtype = rng.choice(["f32", "bf16", "f16"])
    if kind == "plan":
        c = _draw_grid(rng, 48, 160)
        return dict(kind=kind, **c, **_draw_det(rng, c["voxel"], 96, 400), gauss=_logi(rng, 2000, 80000),
                    m0=_logi(rng, 50, 500), m1=_logi(rng, 500, 2000), m2=_logi(rng, 2000, 8000),
                    batch=_logi(rng, 1, 32), dtype=dtype)
    if kind == "autograd":
        c = _draw_grid(rng, 32, 96)
        return dict(kind=kind, **c, **_draw_det(rng, c["voxel"], 64, 200), gauss=_logi(rng, 500, 20000),
                    m0=_logi(rng, 50, 400), m1=rng.choice([0, _logi(rng, 200, 1500)]), m2=0, batch=_logi(rng, 1, 12),
                    dtype="f32")
    if kind in ("vox", "voxgrad"):
        ch = rng.choice([1, 3])
        g = _logi(rng, 2000, 100000) if ch == 1 else _logi(rng, 200, 8000)
        c = dict(kind=kind, **_draw_grid(rng, 48, 200), gauss=g, channels=ch)
        return dict(c, dtype=dtype) if kind == "vox" else c
    if kind == "warp":
        return dict(kind=kind, **_draw_grid(rng, 48, 200), batch=_logi(rng, 1, 32), dtype=dtype,
                    out=rng.choice(["f32", dtype]))
    if kind == "warpgrad":
        return dict(kind=kind, **_draw_grid(rng, 48, 200), batch=_logi(rng, 1, 16), dtype=dtype)
    if kind == "proj":
        c = _draw_grid(rng, 48, 200)
        return dict(kind=kind, **c, **_draw_det(rng, c["voxel"]), batch=_logi(rng, 1, 32), dtype=dtype)
    if kind == "projgrad":
        c = _draw_grid(rng, 48, 200)
        return dict(kind=kind, **c, **_draw_det(rng, c["voxel"]), batch=_logi(rng, 1, 16))
    if kind == "uneven":
        c = _draw_grid(rng, 64, 200)
        return dict(kind=kind, **c, **_draw_det(rng, c["voxel"], 96, 400), items=rng.randint(2, 6),
                    batch=rng.randint(1, 6), dtype=dtype)
    if kind == "eq14":
        c = _draw_grid(rng, 64, 200)
        d = _draw_det(rng, c["voxel"])
        return dict(kind=kind, **c, nu=d["nu"], nv=d["nv"], batch=_logi(rng, 1, 16), crop=rng.choice([16, 24, 32]),
                    dtype=dtype)
    if kind == "stage1":
        c = _draw_grid(rng, 80, 200)
        return dict(kind=kind, **c, **_draw_det(rng, c["voxel"], 128, 512), gauss=_logi(rng, 2000, 100000),
                    batch=_logi(rng, 1, 8), crop=32)
    return dict(kind=kind, **_draw_grid(rng, 48, 200), batch=_logi(rng, 1, 4), dtype=dtype)


# ------------------------------------------------------------------ inputs

class _Rng:
    def __init__(self, seed):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(int(seed) * 7919 + 17)

    def u(self, *shape):
        return torch.rand(shape, generator=self.g, device="cuda")

    def n(self, *shape):
        return torch.randn(shape, generator=self.g, device="cuda")


def _grid(c):
    return (c["nx"], c["ny"], c["nz"], c["voxel"], c["voxel"], c["voxel"])


def _det(c):
    return ops.PmfDetector(c["nu"], c["nv"], c["step"])


def _shape(c):
    return (c["nz"], c["ny"], c["nx"])


def _views(c, r, n):
    """n different views of a 660-view scan."""
    k = torch.randperm(SCAN, generator=r.g, device="cuda")[:n].double()
    th = 2.0 * math.pi * k / SCAN
    co, s, z = torch.cos(th), torch.sin(th), torch.zeros_like(th)
    p = c["pitch"]
    cols = [SAD * co, SAD * s, z, -(SDD - SAD) * co, -(SDD - SAD) * s, z, -p * s, p * co, z, z, z, z + p]
    return torch.stack(cols, 1).contiguous()


def _gaussians(c, r, n, channels, lo, hi, std=None):
    """Centres uniform in the box, scales log-uniform in [lo, hi] voxels, densities U[0, 1] or vectors N(0, std)."""
    ext = torch.tensor([c["nx"], c["ny"], c["nz"]], device="cuda", dtype=torch.float32) * c["voxel"]
    mean = (r.u(n, 3) - 0.5) * ext
    scale = torch.exp(math.log(lo) + (math.log(hi) - math.log(lo)) * r.u(n, 3)) * c["voxel"]
    quat = torch.nn.functional.normalize(r.n(n, 4), dim=1)
    value = r.u(n, channels) if std is None else r.n(n, channels) * std
    return mean.contiguous(), scale.contiguous(), quat.contiguous(), value.contiguous()


def _ref_set(c, r, n):
    lo, hi = (1.0, 4.0) if c["nx"] <= 64 else (0.5, 3.0)
    return _gaussians(c, r, n, 1, lo, hi)


def _mbc_set(c, r, n, std):
    sp = (c["nx"] * c["ny"] * c["nz"] / n) ** (1.0 / 3.0)
    return _gaussians(c, r, n, 3, 0.35 * sp, 0.7 * sp, std)


def _levels(c):
    return [(c[k], s) for k, s in zip(("m0", "m1", "m2"), STDS) if c[k]]


def _smooth(shape, r, sigma):
    """Smooth unit-variance noise: white noise with a Gaussian low-pass of `sigma` voxels."""
    f = torch.fft.rfftn(r.n(*shape))
    k = 0.0
    for d, n in enumerate(shape):
        w = torch.fft.rfftfreq(n, device="cuda") if d == len(shape) - 1 else torch.fft.fftfreq(n, device="cuda")
        k = k + (w ** 2).reshape([-1 if e == d else 1 for e in range(len(shape))])
    x = torch.fft.irfftn(f * torch.exp(-2.0 * (math.pi * sigma) ** 2 * k), s=shape)
    return x / x.std()


def _volume(c, r):
    """A density volume like a voxelized reference set's."""
    return (0.55 + 0.35 * _smooth(_shape(c), r, 1.2)).clamp_min_(0.0)


def _fields(c, r, levels=3):
    """MBC displacement grids [L, 3, nz, ny, nx] in mm, coarse to fine, like the voxelized levels."""
    vox = c["nx"] * c["ny"] * c["nz"]
    out = torch.empty((levels, 3) + _shape(c), device="cuda")
    for l in range(levels):
        sp = (vox / min((500, 2000, 8000)[l] * vox / 4.0e6, vox)) ** (1.0 / 3.0)
        for k in range(3):
            out[l, k] = 0.8 * STDS[l] * _smooth(_shape(c), r, 0.5 * sp)
    return out


def _coeff(r, n, levels):
    """Coefficients of a breathing cycle at n random phases."""
    ph = 2.0 * math.pi * r.u(n, 1, 1)
    return ((0.5 + 0.5 * r.u(1, levels, 3)) * (0.8 + 0.4 * r.u(n, 1, 1))
            * torch.sin(ph + 0.6 * (r.u(1, levels, 3) - 0.5))).contiguous()


def _images(r, n, nv, nu, level):
    """Smooth positive projections of peak about `level` with a little noise."""
    x = torch.nn.functional.interpolate(r.u(n, 1, 7, 9), size=(nv, nu), mode="bicubic", align_corners=True)[:, 0]
    return (level * (0.25 + 0.75 * x.clamp_min(0.0)) + 0.01 * level * r.n(n, nv, nu)).contiguous()


def _residual(r, n, nv, nu):
    """A loss gradient's like: a signed smooth part and pixel noise, over the pixel count."""
    s = torch.nn.functional.interpolate(r.n(n, 1, 9, 11), size=(nv, nu), mode="bicubic", align_corners=True)[:, 0]
    return ((s + 0.2 * r.n(n, nv, nu)) * (20.0 / (n * nv * nu))).contiguous()


def _uneven_items(c):
    """Sizes and view counts of an uneven batch's volumes: each about a quarter smaller than the last."""
    out = []
    for i in range(c["items"]):
        f = 0.8 ** i
        out.append(dict(c, nx=max(16, int(c["nx"] * f)), ny=max(16, int(c["ny"] * f)), nz=max(12, int(c["nz"] * f)),
                        batch=max(1, c["batch"] - 2 * i)))
    return out


def _inputs(c, seed):
    """The case's inputs as device tensors (shared by prepare and exact)."""
    r, kind, B = _Rng(seed), c["kind"], c.get("batch", 1)
    if kind in ("plan", "autograd"):
        ref = _ref_set(c, r, c["gauss"])
        mbc = [_mbc_set(c, r, n, s) for n, s in _levels(c)]
        return dict(ref=ref, mbc=mbc, views=_views(c, r, B), coeff=_coeff(r, B, len(mbc)),
                    meas=_images(r, B, c["nv"], c["nu"], 200.0))
    if kind in ("vox", "voxgrad"):
        gs = _ref_set(c, r, c["gauss"]) if c["channels"] == 1 else _mbc_set(c, r, c["gauss"], 2.0)
        d = None
        if kind == "voxgrad":
            d = torch.stack([_smooth(_shape(c), r, 2.0) + 0.3 * r.n(*_shape(c)) for _ in range(c["channels"])]) * 1e-3
        return dict(gs=gs, d=d)
    if kind in ("warp", "warpgrad", "unfused"):
        dt = DT[c["dtype"]]
        x = dict(V=_volume(c, r).to(dt), E=_fields(c, r).to(dt), coeff=_coeff(r, B, 3))
        if kind != "warp":
            x["d"] = torch.stack([_smooth(_shape(c), r, 2.0) + 0.3 * r.n(*_shape(c)) for _ in range(B)]) * 1e-3
        return x
    if kind == "proj":
        return dict(views=_views(c, r, B), vol=torch.stack([_volume(c, r) for _ in range(B)]).to(DT[c["dtype"]]))
    if kind == "projgrad":
        return dict(views=_views(c, r, B), d=_residual(r, B, c["nv"], c["nu"]))
    if kind == "uneven":
        return [dict(c=k, views=_views(k, r, k["batch"]),
                     vol=torch.stack([_volume(k, r) for _ in range(k["batch"])]).to(DT[c["dtype"]]),
                     d=_residual(r, k["batch"], k["nv"], k["nu"])) for k in _uneven_items(c)]
    if kind == "eq14":
        dt = DT[c["dtype"]]
        E = _fields(c, r)
        E = E * (torch.rsqrt((E.double() ** 2).sum((2, 3, 4), keepdim=True)) * math.sqrt(1.5)).float()
        meas = _images(r, B, c["nv"], c["nu"], 300.0)
        if c["dtype"] == "f16":
            E = E * 64.0  # keeps the components of unit-norm fields clear of the subnormals
        return dict(pred=(meas + 15.0 * torch.nn.functional.interpolate(
            r.n(B, 1, 12, 16), size=(c["nv"], c["nu"]), mode="bicubic", align_corners=True)[:, 0]
            + 2.0 * r.n(B, c["nv"], c["nu"])).contiguous(), meas=meas, V=_volume(c, r).to(dt), E=E.to(dt),
            origin=(torch.tensor([c["nx"], c["ny"], c["nz"]], device="cuda").float() * 0.25).to(torch.int32))
    if kind == "stage1":
        corner = [int(0.3 * c[k]) for k in ("nx", "ny", "nz")]
        return dict(ref=_ref_set(c, r, c["gauss"]), views=_views(c, r, B),
                    meas=_images(r, B, c["nv"], c["nu"], 300.0),
                    centre=pipeline.Stage1Step.crop_centre(_grid(c), corner, c["crop"]).cuda())
    raise ValueError(kind)


# ------------------------------------------------------------------ prepare and run

def prepare(case, seed):
    c, kind = case, case["kind"]
    x = _inputs(c, seed)
    s = dict(c=c, x=x, kind=kind)
    if kind == "plan":
        ref = pmf.Gaussians(*x["ref"], KAPPA)
        mbc = [pmf.Gaussians(*m, KAPPA) for m in x["mbc"]]
        s["plan"] = ops.Plan(_grid(c), _det(c), ref, mbc, c["batch"], DT[c["dtype"]], kind=2, use_graph=True)
        s["Y"] = s["plan"].tensors()["Y"]
        s["Y"].plan = s["plan"]  # a view of the plan's own memory: whoever holds it holds the plan
    elif kind == "autograd":
        for t in [t for m in [x["ref"]] + x["mbc"] for t in m] + [x["coeff"]]:
            t.requires_grad_(True)
    elif kind in ("vox", "voxgrad"):
        s["gs"] = pmf.Gaussians(*x["gs"], KAPPA)
        if kind == "vox":
            cap = int(ops.gs_voxelize_count(_grid(c), s["gs"]) * 1.25) + 4096
            n = ops.gs_voxelize_workspace(_grid(c), s["gs"].n, cap)
            s["ws"] = torch.empty(max(n, 256), dtype=torch.uint8, device="cuda")
            s["out"] = torch.empty((c["channels"],) + _shape(c), dtype=DT[c["dtype"]], device="cuda")
    elif kind == "warp":
        s["out"] = torch.empty((c["batch"],) + _shape(c), dtype=DT[c["out"]], device="cuda")
    elif kind == "stage1":
        step = pipeline.Stage1Step(_grid(c), _det(c), pmf.Gaussians(*x["ref"], KAPPA), c["batch"], 300.0,
                                   tv_size=c["crop"])
        s["step"] = pipeline.GraphedStage1(step, x["views"], x["meas"], x["centre"])
    elif kind == "uneven":
        s["fwd"] = [(_grid(i["c"]), _det(i["c"]), i["views"], i["vol"], False) for i in x]
        s["bwd"] = [(_grid(i["c"]), _det(i["c"]), i["views"], i["d"], False) for i in x]
    return s


def run(s):
    c, x, kind = s["c"], s["x"], s["kind"]
    if kind == "plan":
        p = s["plan"]
        loss = p.step(x["views"], x["coeff"], x["meas"])
        return dict(loss=loss, Y=s["Y"], ref=p.g_ref, mbc=p.g_mbc, coeff=p.d_coeff)
    if kind == "autograd":
        Y, loss = pag.forward_model(_grid(c), _det(c), x["ref"], x["mbc"], x["coeff"], x["views"], x["meas"],
                                    kappa=KAPPA, kind=2, dtype=DT[c["dtype"]])
        leaves = [t for m in [x["ref"]] + x["mbc"] for t in m] + [x["coeff"]]
        return dict(Y=Y.detach(), loss=loss.detach(), grads=torch.autograd.grad(loss, leaves))
    if kind == "vox":
        return ops.gs_voxelize(_grid(c), s["gs"], out=s["out"], ws=s["ws"])
    if kind == "voxgrad":
        return ops.gs_voxelize_backward(_grid(c), s["gs"], x["d"])
    if kind == "warp":
        return ops.warp_combine(_grid(c), x["V"], x["E"], x["coeff"], out=s["out"])
    if kind == "warpgrad":
        return ops.warp_combine_backward(_grid(c), x["V"], x["E"], x["coeff"], x["d"])
    if kind == "proj":
        return ops.conebeam_project(_grid(c), _det(c), x["views"], x["vol"], shared=False)
    if kind == "projgrad":
        return ops.conebeam_project_backward(_grid(c), _det(c), x["views"], x["d"], shared=False)
    if kind == "uneven":
        return dict(Y=ops.conebeam_project_batched(s["fwd"]), dW=ops.conebeam_project_backward_batched(s["bwd"]))
    if kind == "eq14":
        g = _grid(c)
        loss, dY = ops.projection_loss(1, x["pred"], x["meas"])
        ops.projection_dssim(x["pred"], x["meas"], 300.0, weight=0.25, loss=loss, d_pred=dY, accumulate=True)
        tv, dV = ops.tv_loss(g, x["V"], c["crop"], x["origin"], weight=0.05)
        norm, dE = ops.mbc_normality(g, x["E"])
        return dict(loss=loss, dY=dY, tv=tv, dV=dV, norm=norm, dE=dE)
    if kind == "stage1":
        st = s["step"]
        loss, tv = st.run(x["views"], x["meas"], x["centre"])
        return dict(loss=loss, tv=tv, Y=st.step.Y, grads=st.grads)
    g = _grid(c)  # unfused
    D = ops.mbc_combine(g, x["E"], x["coeff"])
    W = ops.warp_volume(g, x["V"], D)
    dV, dD = ops.warp_volume_backward(g, x["V"], D, x["d"])
    dE, dw = ops.mbc_combine_backward(g, x["E"], x["coeff"], dD)
    return dict(D=D, W=W, dV=dV, dE=dE, dw=dw)


# ------------------------------------------------------------------ what a pass cannot do without

def _samples(c, views):
    """March samples of `views` views inside the volume: a coarse grid of rays of 8 views, scaled."""
    n, tot = 8, 0.0
    hx, hy, hz = (0.5 * c[k] * c["voxel"] for k in ("nx", "ny", "nz"))
    u = (np.arange(48) + 0.5) / 48 - 0.5
    a, b = np.meshgrid(u * c["nu"] * c["pitch"], u * c["nv"] * c["pitch"])
    for k in range(n):
        t = 2 * np.pi * (k + 0.3) / n
        d = np.stack([-SDD * np.cos(t) - a * np.sin(t), -SDD * np.sin(t) + a * np.cos(t), b], -1)
        d = d / np.linalg.norm(d, axis=-1, keepdims=True)
        src = np.array([SAD * np.cos(t), SAD * np.sin(t), 0.0])
        with np.errstate(divide="ignore", invalid="ignore"):
            t1, t2 = (-np.array([hx, hy, hz]) - src) / d, (np.array([hx, hy, hz]) - src) / d
        near, far = np.minimum(t1, t2).max(-1), np.maximum(t1, t2).min(-1)
        tot += np.maximum(far - near, 0.0).mean() / c["step"]
    return tot / n * c["nu"] * c["nv"] * views


def _pairs(c, n, lo, hi):
    """(voxel, Gaussian) pairs inside the truncation ellipsoids, scales log-uniform in [lo, hi] voxels."""
    e = (hi - lo) / math.log(hi / lo)
    return n * 4.0 / 3.0 * math.pi * KAPPA ** 3 * e ** 3


def _set_pairs(c, n, channels):
    if channels == 1:
        return _pairs(c, n, *((1.0, 4.0) if c["nx"] <= 64 else (0.5, 3.0)))
    sp = (c["nx"] * c["ny"] * c["nz"] / n) ** (1.0 / 3.0)
    return _pairs(c, n, 0.35 * sp, 0.7 * sp)


def work(c):
    kind, N, B = c["kind"], c["nx"] * c["ny"] * c["nz"], c.get("batch", 1)
    Q = c.get("nu", 0) * c.get("nv", 0)
    el = {"f32": 4, "bf16": 2, "f16": 2}
    if kind in ("plan", "autograd"):
        sets = [(c["gauss"], 1)] + [(n, 3) for n, _ in _levels(c)]
        L = len(sets) - 1
        fl = sum(_set_pairs(c, n, ch) * (40 + 6 * ch) for n, ch in sets)
        fl += _samples(c, B) * (28 + 37) + N * B * (6 * L + 23 + 12 * L + 60)
        par = sum(4 * n * (10 + ch) for n, ch in sets)
        return dict(bytes=2 * par + 2 * 4 * B * Q + 2 * 12 * B * L + 96 * B, flops=fl)
    if kind == "vox":
        n, ch = c["gauss"], c["channels"]
        return dict(bytes=N * ch * el[c["dtype"]] + 4 * n * (10 + ch), flops=_set_pairs(c, n, ch) * (16 + 2 * ch))
    if kind == "voxgrad":
        n, ch = c["gauss"], c["channels"]
        return dict(bytes=4 * N * ch + 8 * n * (10 + ch), flops=_set_pairs(c, n, ch) * (36 + 4 * ch))
    if kind == "warp":
        return dict(bytes=N * (10 * el[c["dtype"]] + B * el[c["out"]]), flops=N * B * (18 + 23))
    if kind == "warpgrad":
        return dict(bytes=N * (10 * el[c["dtype"]] + 4 * B + 40), flops=N * B * (18 + 36 + 36 + 24))
    if kind == "proj":
        return dict(bytes=B * (N * el[c["dtype"]] + 4 * Q), flops=28.0 * _samples(c, B))
    if kind == "projgrad":
        return dict(bytes=4 * B * (N + Q), flops=37.0 * _samples(c, B))
    if kind == "uneven":
        k = _uneven_items(c)
        return dict(bytes=sum(i["batch"] * (i["nx"] * i["ny"] * i["nz"] * (4 + el[c["dtype"]]) + 8 * Q) for i in k),
                    flops=sum(65.0 * _samples(i, i["batch"]) for i in k))
    if kind == "eq14":
        return dict(bytes=12 * B * Q + N * (9 * el[c["dtype"]] + 36) + 4 * N, flops=B * Q * 260 + 30 * N)
    if kind == "stage1":
        lo, hi = (1.0, 4.0) if c["nx"] <= 64 else (0.5, 3.0)
        px = c["voxel"] * SDD / SAD / c["pitch"] * (hi - lo) / math.log(hi / lo)
        pix = min(math.pi * (KAPPA * px) ** 2, float(Q)) * c["gauss"] * B
        return dict(bytes=88 * c["gauss"] + 12 * B * Q, flops=26.0 * pix + 260 * B * Q)
    return dict(bytes=N * ((18 + B + 9) * el[c["dtype"]] + 4 * B + 40), flops=N * B * 110)  # unfused


# ------------------------------------------------------------------ 64-bit results

def _rot64(q):
    q = q / q.norm(dim=1, keepdim=True)
    w, x, y, z = q.unbind(1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1).reshape(-1, 3, 3)


def _vox_chunks(c, gs, limit=3.0e7):
    """(Gaussian range, owner, voxel index, centres) of the voxel boxes, `limit` pairs at a time."""
    n = torch.tensor([c["nx"], c["ny"], c["nz"]], device="cuda", dtype=torch.float64)
    mean, scale, quat = (t.detach().double() for t in gs[:3])
    R = _rot64(quat)
    half = KAPPA * ((R * scale[:, None, :]) ** 2).sum(2).sqrt()
    cen = mean / c["voxel"] + n / 2 - 0.5
    lo = (cen - half / c["voxel"]).floor().sub(1).clamp_min(0).minimum(n).long()
    hi = (cen + half / c["voxel"]).ceil().add(1).clamp_min(-1).minimum(n - 1).long()
    e = (hi - lo + 1).clamp_min(0)
    cnt = e.prod(1)
    run_ = cnt.cumsum(0).cpu().numpy()
    a = 0
    while a < len(run_):
        base = run_[a - 1] if a else 0
        b = max(a + 1, int(np.searchsorted(run_, base + limit)))
        own = torch.repeat_interleave(torch.arange(a, b, device="cuda"), cnt[a:b])
        k = torch.arange(own.numel(), device="cuda") - (cnt[a:b].cumsum(0) - cnt[a:b])[own - a]
        ex, ey = e[own, 0], e[own, 1]
        i, j, l = k % ex + lo[own, 0], (k // ex) % ey + lo[own, 1], k // (ex * ey) + lo[own, 2]
        at = (l * c["ny"] + j) * c["nx"] + i
        xyz = (torch.stack([i, j, l], 1) + 0.5 - n / 2) * c["voxel"]
        yield a, b, own - a, at, xyz
        a = b


def _vox_terms(p, own, xyz):
    """e^{-q/2} of every pair, zero beyond the cutoff; p = (mean, scale, quat) of the chunk in 64 bits."""
    mean, scale, quat = p
    w = torch.einsum("nij,ni->nj", _rot64(quat)[own], xyz - mean[own]) / scale[own]
    q = (w * w).sum(1)
    return torch.exp(-0.5 * q) * (q.detach() <= KAPPA * KAPPA)


def _vox64(c, gs):
    C = gs[3].shape[1]
    out = torch.zeros((C, c["nx"] * c["ny"] * c["nz"]), dtype=torch.float64, device="cuda")
    g64 = [t.detach().double() for t in gs]
    for a, b, own, at, xyz in _vox_chunks(c, gs):
        e = _vox_terms([t[a:b] for t in g64[:3]], own, xyz)
        for k in range(C):
            out[k].index_add_(0, at, e * g64[3][a:b, k][own])
    return out.reshape((C,) + _shape(c))


def _vox64_grad(c, gs, d):
    C, dd = gs[3].shape[1], d.detach().double().reshape(gs[3].shape[1], -1)
    grads = [torch.zeros(t.shape, dtype=torch.float64, device="cuda") for t in gs]
    for a, b, own, at, xyz in _vox_chunks(c, gs, 1.5e7):
        with torch.enable_grad():
            p = [t.detach()[a:b].double().requires_grad_(True) for t in gs]
            e = _vox_terms(p[:3], own, xyz)
            tot = sum((e * p[3][:, k][own] * dd[k][at]).sum() for k in range(C))
            for g, t in zip(grads, torch.autograd.grad(tot, p)):
                g[a:b] = t
    return tuple(grads)


def _warp64(c, V, E, w):
    """One view's warped volume; V [nz,ny,nx], E [L,3,...], w [L,3] in 64 bits (differentiable), and the DVF."""
    D = (w[:, :, None, None, None] * E).sum(0)
    return _pull64(c, V, D), D


def _pull64(c, V, D):
    nz, ny, nx = _shape(c)
    P = torch.nn.functional.pad(V, (1, 2, 1, 2, 1, 2))
    pos = [torch.arange(n, device="cuda", dtype=torch.float64).reshape([-1 if a == k else 1 for a in range(3)])
           + D[2 - k] / c["voxel"] for k, n in enumerate((nz, ny, nx))]
    cell = [p.detach().floor() for p in pos]
    f = [p - q for p, q in zip(pos, cell)]
    ok = torch.ones_like(f[0], dtype=torch.bool)
    idx = []
    for q, n in zip(cell, (nz, ny, nx)):
        ok &= (q >= -1) & (q <= n - 1)
        idx.append((q.clamp(-1, n - 1) + 1).long())
    sy, sz = nx + 3, (nx + 3) * (ny + 3)
    base = idx[0] * sz + idx[1] * sy + idx[2]
    flat, out = P.reshape(-1), 0.0
    for k in range(8):
        dz, dy, dx = k >> 2, (k >> 1) & 1, k & 1
        wt = (f[0] if dz else 1 - f[0]) * (f[1] if dy else 1 - f[1]) * (f[2] if dx else 1 - f[2])
        out = out + flat[base + dz * sz + dy * sy + dx] * wt
    return out * ok


def _march64(c, view, limit=2.5e7):
    """Chunks of one view's rays: (ray slice, cell base in the padded volume, fractions, mask)."""
    v = view.double()
    nu, nv, step, vox = c["nu"], c["nv"], c["step"], c["voxel"]
    n = torch.tensor([c["nx"], c["ny"], c["nz"]], device="cuda", dtype=torch.float64)
    a = torch.arange(nu, device="cuda").double() + 0.5 - nu / 2
    b = torch.arange(nv, device="cuda").double() + 0.5 - nv / 2
    d = v[3:6] - v[0:3] + a[None, :, None] * v[6:9] + b[:, None, None] * v[9:12]
    d = (d / d.norm(dim=2, keepdim=True)).reshape(-1, 3) * (step / vox)
    s = v[0:3] / vox + n / 2 - 0.5
    t1, t2 = (-1.0 - s) / d, (n - s) / d
    lo = torch.minimum(t1, t2).max(1).values.floor().sub(1).clamp_min(0)
    hi = torch.maximum(t1, t2).min(1).values.ceil().add(1)
    cnt = (hi - lo + 1).clamp_min(0)
    m = int(cnt.max().item())
    if m == 0:
        return
    rows = max(1, int(limit / m))
    sy, sz = c["nx"] + 2, (c["nx"] + 2) * (c["ny"] + 2)
    for r0 in range(0, nu * nv, rows):
        r = slice(r0, min(nu * nv, r0 + rows))
        k = lo[r, None] + torch.arange(m, device="cuda").double()
        ok = k <= hi[r, None]
        f, base = [], 0
        for t, st in zip(range(3), (1, sy, sz)):
            u = s[t] + k * d[r, t, None]
            q = u.floor()
            ok &= (q >= -1) & (q <= n[t] - 1)
            f.append(u - q)
            base = base + (q.clamp(-1, float(n[t]) - 1) + 1).long() * st
        yield r, base, f, ok


def _corners64(c, f):
    sy, sz = c["nx"] + 2, (c["nx"] + 2) * (c["ny"] + 2)
    for k in range(8):
        dx, dy, dz = k & 1, (k >> 1) & 1, k >> 2
        yield dz * sz + dy * sy + dx, ((f[0] if dx else 1 - f[0]) * (f[1] if dy else 1 - f[1])
                                       * (f[2] if dz else 1 - f[2]))


def _project64(c, view, vol):
    P = torch.nn.functional.pad(vol.double(), (1, 1, 1, 1, 1, 1)).reshape(-1)
    P = torch.cat([P, P.new_zeros(2 * (c["nx"] + 3) * (c["ny"] + 3))])
    out = torch.zeros(c["nu"] * c["nv"], dtype=torch.float64, device="cuda")
    for r, base, f, ok in _march64(c, view):
        acc = 0.0
        for off, w in _corners64(c, f):
            acc = acc + P[base + off] * w
        out[r] = (acc * ok).sum(1) * c["step"]
    return out.reshape(c["nv"], c["nu"])


def _backproject64(c, view, dY):
    nz, ny, nx = _shape(c)
    n = (nx + 2) * (ny + 2) * (nz + 2)
    acc = torch.zeros(n + 2 * (nx + 3) * (ny + 3), dtype=torch.float64, device="cuda")
    g = dY.double().reshape(-1) * c["step"]
    for r, base, f, ok in _march64(c, view):
        gr = ok * g[r, None]
        for off, w in _corners64(c, f):
            acc.index_add_(0, (base + off).reshape(-1), (gr * w).reshape(-1))
    return acc[:n].reshape(nz + 2, ny + 2, nx + 2)[1:-1, 1:-1, 1:-1].contiguous()


def _warp64_grad(c, V, E, w, d):
    """Gradients of sum_p <W_p, d_p> in V, E and w."""
    gV, gE, gw = torch.zeros_like(V), torch.zeros_like(E), torch.zeros_like(w)
    for p in range(w.shape[0]):
        with torch.enable_grad():
            leaf = [t.detach().requires_grad_(True) for t in (V, E, w[p])]
            W, _ = _warp64(c, *leaf)
            a, b, k = torch.autograd.grad((W * d[p].double()).sum(), leaf)
        gV += a
        gE += b
        gw[p] = k
    return gV, gE, gw


def _window64():
    t = torch.arange(11, device="cuda").double() - 5
    w = torch.exp(-t * t / (2 * 1.5 * 1.5))
    return w / w.sum()


def _dssim64(X, Y, rng_):
    w = _window64()

    def blur(t):
        p = torch.nn.functional.pad(t, (5, 5))
        t = sum(w[k] * p[..., k:k + t.shape[-1]] for k in range(11))
        p = torch.nn.functional.pad(t, (0, 0, 5, 5))
        return sum(w[k] * p[..., k:k + t.shape[-2], :] for k in range(11))

    c1, c2 = (0.01 * rng_) ** 2, (0.03 * rng_) ** 2
    mx, my = blur(X), blur(Y)
    sx, sy, sxy = blur(X * X) - mx * mx, blur(Y * Y) - my * my, blur(X * Y) - mx * my
    return 1 - ((2 * mx * my + c1) * (2 * sxy + c2) / ((mx * mx + my * my + c1) * (sx + sy + c2))).mean()


def _tv64(v):
    return ((v[1:] - v[:-1]).abs().mean() + (v[:, 1:] - v[:, :-1]).abs().mean()
            + (v[:, :, 1:] - v[:, :, :-1]).abs().mean()) / 3


def _splat64_setup(view, gs):
    """Projected 2-D Gaussians of one view: centre (a, b), inverse covariance entries, amplitude, half-widths."""
    v = view.double()
    mean, scale, quat, value = gs
    src, D, du, dv = v[0:3], v[3:6] - v[0:3], v[6:9], v[9:12]
    nrm = torch.linalg.cross(du, dv)
    nrm = nrm / nrm.norm() * torch.sign((nrm * D).sum())
    h = (nrm * D).sum()
    uu, vv, uv = (du * du).sum(), (dv * dv).sum(), (du * dv).sum()
    ut, vt = (vv * du - uv * dv) / (uu * vv - uv * uv), (uu * dv - uv * du) / (uu * vv - uv * uv)
    r = mean - src
    z, ua, vb, L = r @ nrm, r @ ut, r @ vt, r.norm(dim=1)
    a, b = h * ua / z - (ut * D).sum(), h * vb / z - (vt * D).sum()
    Ja = (h / z)[:, None] * (ut - (ua / z)[:, None] * nrm)
    Jb = (h / z)[:, None] * (vt - (vb / z)[:, None] * nrm)
    R = _rot64(quat)
    Ta = torch.einsum("nij,ni->nj", R, Ja) * scale
    Tb = torch.einsum("nij,ni->nj", R, Jb) * scale
    s00, s01, s11 = (Ta * Ta).sum(1), (Ta * Tb).sum(1), (Tb * Tb).sum(1)
    det = s00 * s11 - s01 * s01
    lam = ((torch.einsum("nij,ni->nj", R, r / L[:, None]) / scale) ** 2).sum(1)
    rho = value[:, 0] * torch.sqrt(2 * math.pi / lam)
    return (a, b, s11 / det, -s01 / det, s00 / det, rho), (KAPPA * s00.sqrt(), KAPPA * s11.sqrt())


def _splat64(c, view, gs, d=None, limit=2.0e7):
    """One view's Eq. 9 image, or with d [nv, nu] the gradients of <image, d> in the parameters."""
    g64 = [t.detach().double().requires_grad_(d is not None) for t in gs]
    nu, nv = c["nu"], c["nv"]
    out = torch.zeros(nu * nv, dtype=torch.float64, device="cuda")
    with torch.set_grad_enabled(d is not None):
        p, half = _splat64_setup(view, g64)
    ci, cj = p[0].detach() + 0.5 * nu - 0.5, p[1].detach() + 0.5 * nv - 0.5
    wa, wb = half[0].detach(), half[1].detach()
    i0, i1 = (ci - wa).ceil().sub(1).clamp(0, nu).long(), (ci + wa).floor().add(1).clamp(-1, nu - 1).long()
    j0, j1 = (cj - wb).ceil().sub(1).clamp(0, nv).long(), (cj + wb).floor().add(1).clamp(-1, nv - 1).long()
    ex = (i1 - i0 + 1).clamp_min(0)
    cnt = ex * (j1 - j0 + 1).clamp_min(0)
    run_ = cnt.cumsum(0).cpu().numpy()
    at_p = [torch.zeros_like(t) for t in p]
    k0 = 0
    while k0 < len(run_):
        base = run_[k0 - 1] if k0 else 0
        k1 = max(k0 + 1, int(np.searchsorted(run_, base + limit)))
        own = torch.repeat_interleave(torch.arange(k0, k1, device="cuda"), cnt[k0:k1])
        k = torch.arange(own.numel(), device="cuda") - (cnt[k0:k1].cumsum(0) - cnt[k0:k1])[own - k0]
        i, j = k % ex[own] + i0[own], k // ex[own] + j0[own]
        with torch.set_grad_enabled(d is not None):
            q = [t.detach()[k0:k1].requires_grad_(d is not None) for t in p]
            a, b, K0, K1, K2, rho = (t[own - k0] for t in q)
            da, db = i + 0.5 - nu / 2 - a, j + 0.5 - nv / 2 - b
            qq = K0 * da * da + 2 * K1 * da * db + K2 * db * db
            val = rho * torch.exp(-0.5 * qq) * (qq.detach() <= KAPPA * KAPPA)
            if d is None:
                out.index_add_(0, j * nu + i, val)
            else:
                for t, g in zip(at_p, torch.autograd.grad((val * d.reshape(-1)[j * nu + i]).sum(), q)):
                    t[k0:k1] = g
        k0 = k1
    if d is None:
        return out.reshape(nv, nu)
    return torch.autograd.grad(p, g64, at_p)


def _model64(c, x):
    """The whole L2 step: projections, loss and every gradient."""
    V = _vox64(c, x["ref"])[0]
    E = torch.stack([_vox64(c, m) for m in x["mbc"]])
    w, B = x["coeff"].detach().double(), c["batch"]
    W = [_warp64(c, V, E, w[p])[0] for p in range(B)]
    Y = torch.stack([_project64(c, x["views"][p], W[p]) for p in range(B)])
    diff = Y - x["meas"].double()
    del W
    dW = [_backproject64(c, x["views"][p], 2.0 * diff[p] / diff.numel()) for p in range(B)]
    dV, dE, dw = _warp64_grad(c, V, E, w, dW)
    del dW
    return (Y, (diff * diff).mean(), _vox64_grad(c, x["ref"], dV),
            [_vox64_grad(c, m, dE[l]) for l, m in enumerate(x["mbc"])], dw)


@torch.no_grad()
def exact(case, seed):
    c, kind = case, case["kind"]
    x = _inputs(c, seed)
    if kind in ("plan", "autograd"):
        Y, loss, ref, mbc, dw = _model64(c, x)
        if kind == "plan":
            return dict(loss=loss.reshape(1), Y=Y, ref=ref, mbc=mbc, coeff=dw)
        return dict(Y=Y, loss=loss, grads=[t for m in [ref] + mbc for t in m] + [dw])
    if kind == "vox":
        return _vox64(c, x["gs"])
    if kind == "voxgrad":
        return _vox64_grad(c, x["gs"], x["d"])
    if kind in ("warp", "warpgrad", "unfused"):
        V, E, w = x["V"].double(), x["E"].double(), x["coeff"].double()
        if kind == "warp":
            return torch.stack([_warp64(c, V, E, w[p])[0] for p in range(c["batch"])])
        if kind == "warpgrad":
            return _warp64_grad(c, V, E, w, x["d"])
        # the unfused calls pass the DVF on in the grids' type: the warp and its adjoint see the stored one
        D = torch.stack([(w[p][:, :, None, None, None] * E).sum(0) for p in range(c["batch"])])
        if c["dtype"] != "f32":
            return dict(D=D, W=None, dV=None, dE=None, dw=None)
        gV, gE, gw = _warp64_grad(c, V, E, w, x["d"])
        return dict(D=D, W=torch.stack([_pull64(c, V, D[p]) for p in range(c["batch"])]), dV=gV, dE=gE, dw=gw)
    if kind == "proj":
        return torch.stack([_project64(c, x["views"][p], x["vol"][p]) for p in range(c["batch"])])
    if kind == "projgrad":
        return torch.stack([_backproject64(c, x["views"][p], x["d"][p]) for p in range(c["batch"])])
    if kind == "uneven":
        return dict(Y=[torch.stack([_project64(i["c"], v, o) for v, o in zip(i["views"], i["vol"])]) for i in x],
                    dW=[torch.stack([_backproject64(i["c"], v, o) for v, o in zip(i["views"], i["d"])]) for i in x])
    if kind == "eq14":
        with torch.enable_grad():
            X, V, E = (x[k].double().requires_grad_(True) for k in ("pred", "V", "E"))
            M, D = x["meas"].double(), c["crop"]
            loss = (X - M).abs().mean() + 0.25 * _dssim64(X, M, 300.0)
            o = [int(t) for t in x["origin"].tolist()]
            o = [min(max(k, 0), c[n] - D) for k, n in zip(o, ("nx", "ny", "nz"))]
            tv = 0.05 * _tv64(V[o[2]:o[2] + D, o[1]:o[1] + D, o[0]:o[0] + D])
            norm = (((E * E).sum((2, 3, 4)) - 1) ** 2).mean()
            g = [torch.autograd.grad(t, v)[0] for t, v in ((loss, X), (tv, V), (norm, E))]
        return dict(loss=loss.detach().reshape(1), dY=g[0], tv=tv.detach().reshape(1), dV=g[1],
                    norm=norm.detach().reshape(1), dE=g[2])
    # stage1
    gs, B, D = x["ref"], c["batch"], c["crop"]
    Y = torch.stack([_splat64(c, x["views"][p], gs) for p in range(B)])
    with torch.enable_grad():
        X = Y.clone().requires_grad_(True)
        M = x["meas"].double()
        loss = (X - M).abs().mean() + 0.25 * _dssim64(X, M, 300.0)
        dY = torch.autograd.grad(loss, X)[0]
    grads = [torch.zeros(t.shape, dtype=torch.float64, device="cuda") for t in gs]
    for p in range(B):
        for g, t in zip(grads, _splat64(c, x["views"][p], gs, dY[p])):
            g += t
    cc = dict(c, nx=D, ny=D, nz=D)
    crop = (gs[0] - x["centre"],) + tuple(gs[1:])
    with torch.enable_grad():
        V = _vox64(cc, crop)[0].requires_grad_(True)
        tv = 0.05 * _tv64(V)
        dV = torch.autograd.grad(tv, V)[0]
    for g, t in zip(grads, _vox64_grad(cc, crop, dV[None])):
        g += t
    return dict(loss=loss.detach().reshape(1), tv=tv.detach().reshape(1), Y=Y, grads=grads)
