"""GPU parity of the Stage-1 X-ray rasterizer (Eq. 8-9) against the FP64 oracle
through the C ABI: whole projections at small sizes (several 16x16 tiles,
ragged detector edges, kappa = 3 and no truncation), sampled pixels and
sampled Gaussians' gradients at the paper scale (100,000 Gaussians, 512x384,
32 views), and the edge cases (empty sets, Gaussians behind the source or off
the detector, list overflow, reproducibility).  Forward bar: relative L2
<= 1e-5; gradients <= 1e-3."""
import numpy as np
import pytest
import torch

import oracle
import paper_2503_22139_gb300 as pmf
from synth import Detector, Grid, circular_views, gaussian_set, paper_workload, select_batch, small_workload
from tests.gpu_util import dev, gset, host, pixel_views, rel_l2, views

pytestmark = pytest.mark.gpu

TOL32 = 1e-5
TOLG = 1e-3


def _oracle(det, vw, gs, kappa):
    return oracle.splat(det.nu, det.nv, vw, gs.mean, gs.scale, gs.quat, gs.value, kappa)


@pytest.mark.parametrize("kappa", [3.0, float("inf")])
def test_rasterize_small_workload_matches_oracle(kappa):
    wl = small_workload(with_measured=False)  # 2,000 Gaussians, 8 views of 128^2
    Y = pmf.gs_rasterize(wl.det, views(wl.views), gset(wl.ref, kappa))
    assert rel_l2(host(Y), _oracle(wl.det, wl.views, wl.ref, kappa)) <= TOL32


def _edge_set():
    """Gaussians inside a small volume plus one behind the source of view 0,
    one far off every detector and one straddling the detector edge."""
    grid = Grid(40, 36, 30, 2.0, 2.0, 2.0)
    gs = gaussian_set(np.random.default_rng(21), grid, 300, 0.7, 3.0)
    vw = circular_views(3, 300.0, 450.0, 37, 29, 1.4, 1.4, start=0.3)
    extra = np.array([vw[0, 0:3] * 1.3, [900.0, -900.0, 0.0], [0.0, 0.0, 14.0]], dtype=np.float32)
    gs.mean = np.concatenate([gs.mean, extra]).astype(np.float32)
    gs.scale = np.concatenate([gs.scale, np.full((3, 3), 3.0, np.float32)])
    gs.quat = np.concatenate([gs.quat, np.tile(np.float32([1, 0, 0, 0]), (3, 1))])
    gs.value = np.concatenate([gs.value, np.ones((3, 1), np.float32)])
    return gs, vw, Detector(37, 29, 1.0)


def test_rasterize_ragged_detector_and_edge_gaussians():
    gs, vw, det = _edge_set()
    Y = pmf.gs_rasterize(det, views(vw), gset(gs, 3.0))
    assert rel_l2(host(Y), _oracle(det, vw, gs, 3.0)) <= TOL32


def test_rasterize_empty_and_zero_views():
    gs, vw, det = _edge_set()
    empty = pmf.Gaussians(torch.zeros((0, 3), device="cuda"), torch.zeros((0, 3), device="cuda"),
                          torch.zeros((0, 4), device="cuda"), torch.zeros((0, 1), device="cuda"), 3.0)
    Y = pmf.gs_rasterize(det, views(vw), empty)
    assert torch.equal(Y, torch.zeros_like(Y))
    Y0 = pmf.gs_rasterize(det, views(vw[:0]), gset(gs, 3.0))
    assert Y0.shape == (0, det.nv, det.nu)


def test_rasterize_list_overflow_and_reproducibility():
    """A pair list far too small: every tile scans all Gaussians (same bits,
    counted); and two launches give identical bits (integer pixel sums)."""
    wl = small_workload(with_measured=False)
    g = gset(wl.ref, 3.0)
    vw = views(wl.views)
    a = pmf.gs_rasterize(wl.det, vw, g)
    b = pmf.gs_rasterize(wl.det, vw, g)
    assert torch.equal(a, b)
    pmf.device_counters(reset=True)
    c = pmf.gs_rasterize(wl.det, vw, g, pair_capacity=1)
    assert torch.equal(a, c)
    assert pmf.device_counters()["raster_list_overflow"] > 0
    pmf.device_counters(reset=True)


def test_rasterize_nonfinite_parameter_poisons_its_views():
    gs, vw, det = _edge_set()
    g = gset(gs, 3.0)
    g.scale[5, 1] = float("nan")
    pmf.device_counters(reset=True)
    Y = pmf.gs_rasterize(det, views(vw), g)
    assert torch.isnan(Y).all()
    assert pmf.device_counters()["nonfinite"] > 0
    with pytest.raises(pmf.PmfError):
        pmf.device_status()
    pmf.device_counters(reset=True)


@pytest.mark.parametrize("kappa", [3.0, float("inf")])
def test_rasterize_backward_matches_oracle(kappa):
    gs, vw, det = _edge_set()
    dY = np.random.default_rng(22).normal(size=(len(vw), det.nv, det.nu)).astype(np.float32)
    got = pmf.gs_rasterize_backward(det, views(vw), gset(gs, kappa), dev(dY))
    ref = oracle.splat_backward(det.nu, det.nv, vw, gs.mean, gs.scale, gs.quat, gs.value, dY, kappa)
    for name, a, b in zip(("mean", "scale", "quat", "value"), got, ref):
        assert rel_l2(host(a).reshape(b.shape), b) <= TOLG, name
    # the value gradient is a plain weighted pixel sum
    assert rel_l2(host(got[3]).reshape(-1), ref[3]) <= TOL32


def test_rasterize_backward_accumulates_and_is_reproducible():
    gs, vw, det = _edge_set()
    g = gset(gs, 3.0)
    dY = dev(np.random.default_rng(23).normal(size=(len(vw), det.nv, det.nu)))
    a = pmf.gs_rasterize_backward(det, views(vw), g, dY)
    b = pmf.gs_rasterize_backward(det, views(vw), g, dY)
    for x, y in zip(a, b):
        assert torch.equal(x, y)
    base = [torch.full_like(t, 0.5) for t in a]
    pmf.gs_rasterize_backward(det, views(vw), g, dY, grads=base, accumulate=True)
    for x, y in zip(base, a):
        assert torch.allclose(x, y + 0.5, rtol=0, atol=1e-5 * (1 + float(y.abs().max())))


@pytest.fixture(scope="module")
def paper():
    wl = paper_workload(p=660)
    idx = select_batch(wl.p, 32, 0)
    return wl, wl.views[idx]


def test_rasterize_paper_scale_sampled_pixels(paper):
    """The benchmark's Stage-1 launch (100,000 Gaussians, 32 views of 512x384):
    64 sampled pixels against the oracle, one 1x1 view per pixel."""
    wl, vw = paper
    Y = host(pmf.gs_rasterize(wl.det, views(vw), gset(wl.ref, wl.kappa)))
    rng = np.random.default_rng(24)
    pix = [(int(rng.integers(0, 32)), int(rng.integers(0, wl.det.nv)), int(rng.integers(0, wl.det.nu)))
           for _ in range(64)]
    ref = oracle.splat(1, 1, pixel_views(vw, wl.det.nu, wl.det.nv, pix), wl.ref.mean, wl.ref.scale, wl.ref.quat,
                       wl.ref.value, wl.kappa)[:, 0, 0]
    got = np.array([Y[p, b, a] for p, b, a in pix])
    assert rel_l2(got, ref) <= TOL32


def test_rasterize_paper_scale_gradients(paper):
    """The adjoint at the paper scale: <dY, Y> = sum_g rho_g dL/drho_g (Y is
    linear in the densities) over the whole batch, and 48 sampled Gaussians'
    gradients against the oracle (a Gaussian's gradient depends only on its own
    parameters and dY)."""
    wl, vw = paper
    g = gset(wl.ref, wl.kappa)
    Y = pmf.gs_rasterize(wl.det, views(vw), g)
    dY = torch.randn(Y.shape, device="cuda", generator=torch.Generator("cuda").manual_seed(25))
    grads = pmf.gs_rasterize_backward(wl.det, views(vw), g, dY)
    lhs = float((dY.double() * Y.double()).sum())
    rhs = float((g.value.double().reshape(-1) * grads[3].double().reshape(-1)).sum())
    assert rhs == pytest.approx(lhs, rel=1e-5)
    sel = np.random.default_rng(26).choice(wl.ref.mean.shape[0], 48, replace=False)
    ref = oracle.splat_backward(wl.det.nu, wl.det.nv, vw, wl.ref.mean[sel], wl.ref.scale[sel], wl.ref.quat[sel],
                                wl.ref.value[sel], host(dY), wl.kappa)
    for name, a, b in zip(("mean", "scale", "quat", "value"), grads, ref):
        assert rel_l2(host(a)[sel].reshape(b.shape), b) <= TOLG, name


@pytest.mark.parametrize("nu", [37, 40])
def test_rasterize_adjoint_run_blocks(nu):
    """The render's and the adjoint's pixel blocks at their extremes: runs of one
    pixel to the whole row, Gaussians far narrower than a pixel (whose
    exponential a few pixels out underflows) and wider than the detector, on
    image rows that are and are not 16-byte multiples, against the oracle."""
    grid = Grid(24, 20, 16, 2.0, 2.0, 2.0)
    rng = np.random.default_rng(61)
    gs = gaussian_set(rng, grid, 60, 0.5, 3.0)
    gs.scale[:20] = np.float32(0.05)  # 0.05 mm: a few hundredths of a pixel
    gs.scale[20:24] = np.float32(40.0)  # wider than the detector
    vw = circular_views(2, 300.0, 450.0, nu, 29, 1.4, 1.4, start=0.4)
    det = Detector(nu, 29, 1.0)
    Y = pmf.gs_rasterize(det, views(vw), gset(gs, 3.0))
    assert rel_l2(host(Y), _oracle(det, vw, gs, 3.0)) <= TOL32
    dY = rng.normal(size=(2, 29, nu)).astype(np.float32)
    got = pmf.gs_rasterize_backward(det, views(vw), gset(gs, 3.0), dev(dY))
    ref = oracle.splat_backward(det.nu, det.nv, vw, gs.mean, gs.scale, gs.quat, gs.value, dY, 3.0)
    for name, a, b in zip(("mean", "scale", "quat", "value"), got, ref):
        assert rel_l2(host(a), np.asarray(b).reshape(tuple(a.shape))) <= TOLG, name


@pytest.mark.parametrize("kappa", [3.0, float("inf")])
@pytest.mark.parametrize("ratio", [10.0, 30.0, 100.0])
def test_rasterize_keeps_flat_rotated_gaussians(ratio, kappa):
    """The render drops pixel blocks that a projected ellipse cannot reach; a flat
    one's fp32 quadratic form loses digits, which the drop must allow for.  With
    u = 2^-24 the elements of Sigma^ are good to 30 u of its largest (three-term
    sums of products good to 10 u), so the form and its inverse to 100 u cond q;
    p^ to an ulp adds 2 |K d| of it.  Every pixel lies between the sums with q
    that much larger and smaller, and rho^ a thousandth (40 u ratio, at most
    2.4e-4), give or take the pixel sums' 2^-21 rounding; with and without lists."""
    rng = np.random.default_rng(62 + int(ratio))
    G, nu, nv = 60, 40, 29
    wide = np.exp(rng.uniform(np.log(4.0), np.log(14.0), G))
    scale = np.stack([wide, np.where(np.arange(G) % 2, wide / ratio, wide), wide / ratio], 1).astype(np.float32)
    mean, quat = rng.uniform(-12.0, 12.0, (G, 3)).astype(np.float32), rng.normal(size=(G, 4)).astype(np.float32)
    value = rng.uniform(0.5, 1.0, (G, 1)).astype(np.float32)
    vw, det = circular_views(2, 300.0, 450.0, nu, nv, 1.4, 1.4, start=0.4), Detector(nu, nv, 1.0)
    g = pmf.Gaussians(dev(mean), dev(scale), dev(quat), dev(value), kappa)
    got = pmf.gs_rasterize(det, views(vw), g)
    assert torch.equal(got, pmf.gs_rasterize(det, views(vw), g, pair_capacity=1))
    xa, xb = np.meshgrid(np.arange(nu) + 0.5 - nu / 2, np.arange(nv) + 0.5 - nv / 2)
    u, k2 = 2.0 ** -24, kappa * kappa
    for p in range(2):
        lower, upper, top = np.zeros((nv, nu)), np.zeros((nv, nu)), 0.0
        for i in range(G):
            pa, pb, s00, s01, s11, rho = oracle.splat_params(vw[p], mean[i], scale[i], quat[i], value[i, 0])[:6]
            S = np.array([[s00, s01], [s01, s11]])
            K, ev = np.linalg.inv(S), np.linalg.eigvalsh(S)
            d = np.stack([xa - pa, xb - pb], -1)
            Kd = d @ K
            q = (Kd * d).sum(-1)
            dq = 100 * u * ev[1] / ev[0] * q + 2 * np.linalg.norm(Kd, axis=-1) * 2 * u * (abs(pa) + abs(pb) + nu)
            lower += 0.999 * rho * np.where(q + dq <= k2, np.exp(-0.5 * (q + dq)), 0.0)
            upper += 1.001 * rho * np.where(q - dq <= k2, np.exp(-0.5 * np.maximum(q - dq, 0.0)), 0.0)
            top = max(top, rho)
        y, tol = host(got)[p], top * G * 2.0 ** -21 + 1e-6 * upper
        assert lower.sum() > 10.0 and np.all(y >= lower - tol) and np.all(y <= upper + tol)
