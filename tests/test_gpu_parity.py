"""GPU parity: every stage of the CUDA path (called through the C ABI) against
the FP64 oracle on the same seeded inputs.  FP32 bar: relative L2 <= 1e-5
(tighter where the arithmetic allows); gradients <= 1e-3 relative."""
import numpy as np
import pytest
import torch

import oracle
import paper_2503_22139_gb300 as pmf
from synth import Detector, Grid, circular_views, small_workload, fd_subproblem, gaussian_set, mbc_levels
from tests import oracle_chain
from tests.gpu_util import assert_voxels_match, dev, gset, host, pixel_views, rel_l2, tie_band, views

pytestmark = pytest.mark.gpu

TOL32 = 1e-5


@pytest.fixture(scope="module", autouse=True)
def _lib_loaded(gpu_lib):
    return gpu_lib


def _rand_gaussians(seed, grid, G, lo, hi, C, std=None):
    return gaussian_set(np.random.default_rng(seed), grid, G, lo, hi, channels=C, value_std=std)


# ------------------------------------------------------------- voxelizer

@pytest.mark.parametrize("kappa", [3.0, float("inf")])
def test_voxelize_ragged_grid(kappa):
    grid = Grid(13, 11, 9, 2.0, 2.5, 3.0)  # several 8^3 tiles with ragged edges
    gs = _rand_gaussians(1, grid, 60, 0.7, 3.0, 1)
    got = host(pmf.gs_voxelize(grid, gset(gs, kappa)))
    ref = oracle.voxelize(grid, gs.mean, gs.scale, gs.quat, gs.value, kappa)
    amb, _ = tie_band(grid, gs, kappa)
    assert_voxels_match(got, ref, amb, TOL32)


@pytest.mark.parametrize("kappa", [3.0, 5.0])
def test_voxelize_small_workload_reference_and_mbc(kappa):
    """At the workloads' kappa = 3 the voxels outside the binary32 tie band hold
    1e-5 and the rest their tie mass; the number of pairs in the band and of
    voxels where a tie actually went the other way are printed.  At kappa = 5
    a flipped tie moves a voxel by at most max|value| e^{-12.5}, so every voxel
    of the volume, ties included, holds 1e-5."""
    wl = small_workload(with_measured=False)
    for gs in (wl.ref, wl.mbc[0]):
        got = host(pmf.gs_voxelize(wl.grid, gset(gs, kappa)))
        ref = oracle.voxelize(wl.grid, gs.mean, gs.scale, gs.quat, gs.value, kappa)
        amb, npairs = tie_band(wl.grid, gs, kappa)
        assert got.shape == (gs.channels,) + wl.grid.shape
        sure, flipped = assert_voxels_match(got, ref, amb, TOL32)
        print(f"kappa {kappa} C={gs.channels}: all-voxel rel-L2 {rel_l2(got, ref):.2e}, {npairs} pairs in the tie "
              f"band, {int((amb > 0).sum())} voxels touched, {flipped} decided the other way")
        assert sure > (0.999 if kappa == 3.0 else 0.99)
        if kappa == 5.0:
            assert rel_l2(got, ref) <= TOL32  # all voxels, ties included


@pytest.mark.parametrize("tile", [(16, 8, 8), (8, 8, 4), (16, 8, 4)])
@pytest.mark.parametrize("C,kappa", [(1, 3.0), (3, 3.0), (3, float("inf"))])
def test_voxelize_bin_tiles_give_the_same_bits(tile, C, kappa):
    """Every bin tile sums the same exactly-rounded terms, so the volume is the
    default tile's bit for bit -- on a ragged grid, through the pair lists and
    through the overflow path that scans every Gaussian -- and it matches the
    oracle like the default."""
    grid = Grid(37, 22, 13, 2.0, 2.0, 2.5)
    gs = _rand_gaussians(5 + C, grid, 120, 0.7, 3.5, C, 2.0 if C == 3 else None)
    g = gset(gs, kappa)
    base = pmf.gs_voxelize(grid, g)
    got = pmf.gs_voxelize_tiled(grid, g, tile)
    assert torch.equal(base, got)
    assert torch.equal(base, pmf.gs_voxelize(grid, g, tile=tile, pair_capacity=11))
    ref = oracle.voxelize(grid, gs.mean, gs.scale, gs.quat, gs.value, kappa)
    amb, _ = tie_band(grid, gs, kappa)
    assert_voxels_match(host(got), ref, amb, TOL32)
    # the pair count depends on the tile: a tile made of whole 8^3 tiles lists
    # each Gaussian in at most as many tiles, one that subdivides 8^3 in at least
    n8 = pmf.gs_voxelize_count(grid, g)
    nt = pmf.gs_voxelize_tiled_count(grid, g, tile)
    if all(t >= 8 for t in tile):
        assert nt <= n8
    elif all(t <= 8 for t in tile):
        assert nt >= n8
    assert nt > 0


def test_voxelize_list_overflow_falls_back_correctly():
    """A pair capacity far below the overlap count routes tiles through the
    scan-everything path; the result must not change by a bit."""
    grid = Grid(24, 20, 17, 2.0, 2.0, 2.0)
    gs = gset(_rand_gaussians(2, grid, 300, 0.7, 4.0, 3, 2.0), 3.0)
    full = pmf.gs_voxelize(grid, gs)
    small = pmf.gs_voxelize(grid, gs, pair_capacity=37)
    zero = pmf.gs_voxelize(grid, gs, pair_capacity=0)
    torch.testing.assert_close(full, small, rtol=0, atol=0)
    torch.testing.assert_close(full, zero, rtol=0, atol=0)


def test_voxelize_edge_cases():
    grid = Grid(9, 8, 7, 2.0, 2.0, 2.0)
    empty = pmf.Gaussians(dev(np.zeros((0, 3))), dev(np.ones((0, 3))), dev(np.ones((0, 4))), dev(np.zeros((0, 1))))
    assert float(pmf.gs_voxelize(grid, empty).abs().max()) == 0.0
    # entirely outside the volume
    far = pmf.Gaussians(dev([[500.0, 0, 0]]), dev([[1.0, 1, 1]]), dev([[1.0, 0, 0, 0]]), dev([[1.0]]), 3.0)
    assert float(pmf.gs_voxelize(grid, far).abs().max()) == 0.0
    # one voxel grid
    g1 = Grid(1, 1, 1, 1.0, 1.0, 1.0)
    one = pmf.Gaussians(dev([[0.0, 0, 0]]), dev([[1.0, 1, 1]]), dev([[1.0, 0, 0, 0]]), dev([[2.0]]), 3.0)
    assert float(pmf.gs_voxelize(g1, one).item()) == pytest.approx(2.0, rel=1e-7)


def test_voxelize_is_bit_reproducible():
    wl = small_workload(with_measured=False)
    gs = gset(wl.mbc[0], wl.kappa)
    a = pmf.gs_voxelize(wl.grid, gs)
    b = pmf.gs_voxelize(wl.grid, gs)
    assert torch.equal(a, b)


@pytest.mark.parametrize("C,kappa", [(1, float("inf")), (3, float("inf")), (1, 3.0), (3, 2.5)])
def test_voxelize_backward_matches_oracle(C, kappa):
    grid = Grid(12, 10, 11, 2.0, 2.0, 2.0)
    gs = _rand_gaussians(3 + C, grid, 40, 0.8, 3.0, C, 2.0 if C == 3 else None)
    rng = np.random.default_rng(7)
    d_out = rng.normal(size=(C,) + grid.shape).astype(np.float32)
    got = pmf.gs_voxelize_backward(grid, gset(gs, kappa), dev(d_out))
    ref = oracle.voxelize_backward(grid, gs.mean, gs.scale, gs.quat, gs.value, d_out, kappa)
    for name, g_, r_ in zip(("mean", "scale", "quat", "value"), got, ref):
        assert rel_l2(host(g_), r_) <= 1e-4, name


@pytest.mark.parametrize("C", [2, 4])
def test_voxelize_two_and_four_channels(C):
    """The two- and four-channel forms against the oracle: the forward on the
    default and the widest bin tile (same bits; at four channels its staged
    records need more than 48 KB of shared memory) and the adjoint."""
    grid = Grid(21, 18, 15, 2.0, 2.0, 2.0)
    gs = _rand_gaussians(40 + C, grid, 80, 0.7, 3.0, C, 1.5)
    g = gset(gs, 3.0)
    base = pmf.gs_voxelize(grid, g)
    assert torch.equal(base, pmf.gs_voxelize_tiled(grid, g, (16, 8, 8)))
    ref = oracle.voxelize(grid, gs.mean, gs.scale, gs.quat, gs.value, 3.0)
    amb, _ = tie_band(grid, gs, 3.0)
    assert_voxels_match(host(base), ref, amb, TOL32)
    d_out = np.random.default_rng(60 + C).normal(size=(C,) + grid.shape).astype(np.float32)
    got = pmf.gs_voxelize_backward(grid, gset(gs, float("inf")), dev(d_out))
    refb = oracle.voxelize_backward(grid, gs.mean, gs.scale, gs.quat, gs.value, d_out, float("inf"))
    for name, g_, r_ in zip(("mean", "scale", "quat", "value"), got, refb):
        assert rel_l2(host(g_), r_) <= 1e-4, name


def test_voxelize_backward_vector_loads_give_the_same_bits():
    """With several channels on 16-byte rows the adjoint reads the upstream
    gradient 16 bytes at a time; the same values at a pointer off the 16-byte
    boundary take scalar loads.  The voxels visited and their order are the
    same, so the gradients are too, bit for bit, and they match the oracle."""
    grid = Grid(24, 14, 11, 2.0, 2.0, 2.0)
    gs = _rand_gaussians(71, grid, 60, 0.8, 4.0, 3, 2.0)
    d_out = np.random.default_rng(72).normal(size=(3,) + grid.shape).astype(np.float32)
    aligned = dev(d_out)
    buf = torch.zeros(aligned.numel() + 1, device="cuda")
    buf[1:] = aligned.reshape(-1)
    shifted = buf[1:].view(aligned.shape)  # 4 bytes past a 16-byte boundary
    assert shifted.data_ptr() % 16 != 0 and aligned.data_ptr() % 16 == 0
    g = gset(gs, 3.0)
    got_v = pmf.gs_voxelize_backward(grid, g, aligned)
    got_s = pmf.gs_voxelize_backward(grid, g, shifted)
    for a, b in zip(got_v, got_s):
        assert torch.equal(a, b)
    ref = oracle.voxelize_backward(grid, gs.mean, gs.scale, gs.quat, gs.value, d_out, 3.0)
    for name, g_, r_ in zip(("mean", "scale", "quat", "value"), got_v, ref):
        assert rel_l2(host(g_), r_) <= 1e-4, name


def test_voxelize_backward_accumulates():
    grid = Grid(8, 8, 8, 2.0, 2.0, 2.0)
    gs = gset(_rand_gaussians(9, grid, 10, 1.0, 2.0, 1), 3.0)
    d_out = dev(np.random.default_rng(1).normal(size=(1,) + grid.shape))
    a = pmf.gs_voxelize_backward(grid, gs, d_out)
    b = pmf.gs_voxelize_backward(grid, gs, d_out, grads=tuple(t.clone() for t in a), accumulate=True)
    for x, y in zip(a, b):
        torch.testing.assert_close(2 * x, y, rtol=1e-6, atol=1e-6)


# --------------------------------------------------- combine and warp

def _mbc_and_ref(grid, seed, L=3, P=5):
    rng = np.random.default_rng(seed)
    V = rng.random(grid.shape).astype(np.float32)
    E = rng.normal(0, 2.0, (L, 3) + grid.shape).astype(np.float32)
    w = rng.uniform(-1, 1, (P, L, 3)).astype(np.float32)
    return V, E, w


def test_combine_and_warp_match_oracle():
    grid = Grid(21, 17, 13, 2.0, 2.0, 2.0)
    V, E, w = _mbc_and_ref(grid, 11)
    D = pmf.mbc_combine(grid, dev(E), dev(w))
    Dref = oracle.combine(E, w)
    assert rel_l2(host(D), Dref) <= 1e-6
    W = pmf.warp_volume(grid, dev(V), D)
    Wref = oracle.warp(grid, V, host(D))
    assert rel_l2(host(W), Wref) <= TOL32
    Wf = pmf.warp_combine(grid, dev(V), dev(E), dev(w))
    assert rel_l2(host(Wf), oracle.warp(grid, V, Dref)) <= TOL32


@pytest.mark.parametrize("L,dt", [(2, torch.bfloat16), (3, torch.float16), (6, torch.bfloat16)])
def test_warp_combine_fp32_output_from_reduced_grids(L, dt):
    """warp_combine_mixed: bf16 / fp16 V and E, fp32 W (the 8x8x4 tile kernel
    for L <= 4, the per-voxel kernel above).  W is the fp32 warp of the stored
    grids' values, and rounding it to the grids' format gives the same-format
    entry point's output bit for bit (both round the same fp32 sum once)."""
    grid = Grid(37, 11, 9, 2.0, 2.0, 2.0)
    V, E, w = _mbc_and_ref(grid, 50 + L, L=L, P=3)
    Vd, Ed = dev(V).to(dt), dev(E).to(dt)
    W32 = torch.empty((3,) + grid.shape, device="cuda")
    pmf.warp_combine(grid, Vd, Ed, dev(w), out=W32)
    Vq, Eq = host(Vd).astype(np.float64), host(Ed).astype(np.float64)
    assert rel_l2(host(W32), oracle.warp(grid, Vq, oracle.combine(Eq, w))) <= TOL32
    Wn = pmf.warp_combine(grid, Vd, Ed, dev(w))
    assert Wn.dtype == dt and torch.equal(W32.to(dt), Wn)


def test_zero_dvf_warp_is_bitwise_identity():
    grid = Grid(9, 8, 7, 2.0, 2.0, 2.0)
    V = dev(np.random.default_rng(3).random(grid.shape))
    W = pmf.warp_volume(grid, V, torch.zeros((2, 3) + grid.shape, device="cuda"))
    assert torch.equal(W[0], V) and torch.equal(W[1], V)


def test_combine_and_warp_backward_match_oracle():
    grid = Grid(19, 15, 12, 2.0, 2.0, 2.0)
    V, E, w = _mbc_and_ref(grid, 12, L=3, P=4)
    rng = np.random.default_rng(13)
    dW = rng.normal(size=(4,) + grid.shape).astype(np.float32)
    Dref = oracle.combine(E, w)
    dV_ref, dD_ref = oracle.warp_backward(grid, V, Dref, dW)
    dE_ref, dw_ref = oracle.combine_backward(E, w, dD_ref)
    D = pmf.mbc_combine(grid, dev(E), dev(w))
    dV, dD = pmf.warp_volume_backward(grid, dev(V), D, dev(dW))
    assert rel_l2(host(dV), dV_ref) <= TOL32
    assert rel_l2(host(dD), dD_ref) <= 1e-4
    dE, dw = pmf.mbc_combine_backward(grid, dev(E), dev(w), dev(dD_ref.astype(np.float32)))
    dE_r2, dw_r2 = oracle.combine_backward(E, w, dD_ref.astype(np.float32))
    assert rel_l2(host(dE), dE_r2) <= 1e-6
    assert rel_l2(host(dw), dw_r2) <= 1e-5
    fdV, fdE, fdw = pmf.warp_combine_backward(grid, dev(V), dev(E), dev(w), dev(dW))
    assert rel_l2(host(fdV), dV_ref) <= TOL32
    assert rel_l2(host(fdE), dE_ref) <= 1e-4
    assert rel_l2(host(fdw), dw_ref) <= 1e-4


@pytest.mark.parametrize("L", [1, 2, 4])
def test_fused_warp_tile_kernels_every_level_count(L):
    """The tile kernels (8x8x4 forward, 8x16x4 adjoint) are instantiated per level count (L <= 4); each
    reduces its 3 L coefficient-gradient values per view across the warp by
    halving exchange, whose slot layout depends on 3 L.  Forward and adjoint of
    every instance against the oracle on a ragged grid."""
    grid = Grid(35, 9, 7, 2.0, 2.0, 2.0)
    V, E, w = _mbc_and_ref(grid, 90 + L, L=L, P=6)
    D = oracle.combine(E, w)
    W = host(pmf.warp_combine(grid, dev(V), dev(E), dev(w)))
    assert rel_l2(W, oracle.warp(grid, V, D)) <= TOL32
    dW = np.random.default_rng(95 + L).normal(size=(6,) + grid.shape).astype(np.float32)
    dV_ref, dD_ref = oracle.warp_backward(grid, V, D, dW)
    dE_ref, dw_ref = oracle.combine_backward(E, w, dD_ref)
    dV, dE, dw = pmf.warp_combine_backward(grid, dev(V), dev(E), dev(w), dev(dW))
    assert rel_l2(host(dV), dV_ref) <= TOL32
    assert rel_l2(host(dE), dE_ref) <= 1e-4
    assert rel_l2(host(dw), dw_ref) <= 1e-4


def test_fused_warp_displacements_beyond_the_staged_halo():
    """MBC vectors of 12 mm std on 2 mm voxels: many displaced samples leave
    the tile's staged 4-voxel halo (the kernels then read and scatter through
    global memory), some leave the grid, and one voxel's displacement is 10^30
    mm (outside the range of the fast floor; zero padding).  Forward and
    adjoint still match the oracle."""
    grid = Grid(45, 13, 10, 2.0, 2.0, 2.0)
    rng = np.random.default_rng(71)
    L, P = 2, 3
    V = rng.random(grid.shape).astype(np.float32)
    E = rng.normal(0, 12.0, (L, 3) + grid.shape).astype(np.float32)
    E[0, 1, 4, 6, 20] = 1e30
    w = rng.uniform(-1, 1, (P, L, 3)).astype(np.float32)
    w[:, 0, 1] = np.abs(w[:, 0, 1]) + 0.1
    D = oracle.combine(E, w)
    far = np.abs(D) / 2.0 > 4.0
    assert far.any(axis=1).mean() > 0.2
    W = host(pmf.warp_combine(grid, dev(V), dev(E), dev(w)))
    Wref = oracle.warp(grid, V, D)
    assert np.all(W[:, 4, 6, 20] == 0.0) and np.all(Wref[:, 4, 6, 20] == 0.0)
    assert rel_l2(W, Wref) <= TOL32
    dW = rng.normal(size=(P,) + grid.shape).astype(np.float32)
    dW[:, 4, 6, 20] = 0.0  # the 10^30 voxel has no finite DVF gradient to compare
    dV_ref, dD_ref = oracle.warp_backward(grid, V, D, dW)
    dE_ref, dw_ref = oracle.combine_backward(E, w, dD_ref)
    dV, dE, dw = pmf.warp_combine_backward(grid, dev(V), dev(E), dev(w), dev(dW))
    assert rel_l2(host(dV), dV_ref) <= TOL32
    assert rel_l2(host(dE), dE_ref) <= 1e-4
    assert rel_l2(host(dw), dw_ref) <= 1e-4


def test_warp_backward_is_bit_reproducible():
    grid = Grid(19, 15, 12, 2.0, 2.0, 2.0)
    V, E, w = _mbc_and_ref(grid, 14, L=3, P=4)
    dW = dev(np.random.default_rng(15).normal(size=(4,) + grid.shape))
    a = pmf.warp_combine_backward(grid, dev(V), dev(E), dev(w), dW)
    b = pmf.warp_combine_backward(grid, dev(V), dev(E), dev(w), dW)
    for x, y in zip(a, b):
        assert torch.equal(x, y)


# ------------------------------------------------------------ projector

@pytest.mark.parametrize("nu,nv", [(37, 23), (16, 16)])
def test_project_ragged_detector(nu, nv):
    grid = Grid(20, 18, 14, 2.0, 2.0, 2.5)
    rng = np.random.default_rng(21)
    vol = rng.random((3,) + grid.shape).astype(np.float32)
    vw = circular_views(3, 400.0, 600.0, nu, nv, 1.8, 1.9, start=0.37)
    got = host(pmf.conebeam_project(grid, Detector(nu, nv, 1.0), views(vw), dev(vol)))
    ref = oracle.project(grid, nu, nv, 1.0, vw, vol)
    assert rel_l2(got, ref) <= TOL32


@pytest.mark.parametrize("shared", [False, True])
def test_project_bulk_copy_staging_equals_plain_staging(shared):
    """fp32 volumes whose rows are whole 16-byte lines get their shared-memory
    boxes by bulk tensor copies; bf16 volumes by plain loads.  On values that
    bf16 holds exactly both forms must give the same projections bit for bit
    (the samples and their order do not depend on how the box was filled),
    and no bulk copy may time out."""
    grid = Grid(48, 44, 36, 2.0, 2.0, 2.0)
    P = 4
    vol = np.random.default_rng(23).random((P,) + grid.shape).astype(np.float32)
    vb = dev(vol).to(torch.bfloat16)
    src = vb[0] if shared else vb
    vw = circular_views(P, 500.0, 750.0, 70, 54, 2.2, 2.2, start=0.2)
    det = Detector(70, 54, 1.0)
    pmf.device_counters(reset=True)
    y32 = pmf.conebeam_project(grid, det, views(vw), src.float(), shared=shared)
    y16 = pmf.conebeam_project(grid, det, views(vw), src, shared=shared)
    assert torch.equal(y32, y16)
    assert pmf.device_counters()["timeout"] == 0
    pmf.device_status()
    ref = oracle.project(grid, 70, 54, 1.0, vw, host(src), shared=shared)
    assert rel_l2(host(y32), ref) <= TOL32


def test_bulk_copy_wait_timeout_is_reported_and_recovers():
    """The failure path of the bulk-copy projector's bounded wait, without a
    fault: the test hook arms each chunk's mbarrier but issues no copy, so every
    CTA that stages a box gives up after its short limit with nothing in flight.
    Its pixels are NaN (the others equal a clean launch), the timeout counter
    rises and pmf_device_status reports PMF_ETIMEOUT; once the hook is off, the
    next launch equals a clean one bit for bit and the status is OK again."""
    grid = Grid(48, 44, 36, 2.0, 2.0, 2.0)
    P = 3
    vol = dev(np.random.default_rng(24).random(grid.shape).astype(np.float32))
    vw = views(circular_views(P, 500.0, 750.0, 70, 54, 2.2, 2.2, start=0.3))
    det = Detector(70, 54, 1.0)
    pmf.device_counters(reset=True)
    clean = pmf.conebeam_project(grid, det, vw, vol, shared=True)
    pmf.device_status()
    try:
        pmf.ops.pmf_debug_stall_bulk_copies(True)
        stalled = pmf.conebeam_project(grid, det, vw, vol, shared=True)
        torch.cuda.synchronize()
    finally:
        pmf.ops.pmf_debug_stall_bulk_copies(False)
    # a CTA that stages a box times out and writes NaN to all its pixels; one
    # whose every chunk takes the global-gather fallback computes as usual
    nan = torch.isnan(stalled)
    assert bool(torch.equal(stalled[~nan], clean[~nan]))
    hit = clean != 0
    assert float(nan[hit].float().mean()) > 0.5
    assert pmf.device_counters()["timeout"] > 0
    with pytest.raises(pmf.PmfError, match="ETIMEOUT"):
        pmf.device_status()
    pmf.device_counters(reset=True)
    again = pmf.conebeam_project(grid, det, vw, vol, shared=True)
    assert torch.equal(again, clean)
    assert pmf.device_counters()["timeout"] == 0
    pmf.device_status()


def test_project_small_workload_voxelized_reference():
    wl = small_workload(with_measured=False)
    V = pmf.gs_voxelize(wl.grid, gset(wl.ref, wl.kappa))[0]
    Vh = host(V)
    got = host(pmf.conebeam_project(wl.grid, wl.det, views(wl.views), V, shared=True))
    ref = oracle.project(wl.grid, wl.det.nu, wl.det.nv, wl.det.step_mm, wl.views, Vh)
    assert rel_l2(got, ref) <= TOL32


def test_project_shared_volume_and_rays_that_miss():
    grid = Grid(16, 16, 16, 2.0, 2.0, 2.0)
    vol = np.random.default_rng(4).random(grid.shape).astype(np.float32)
    vw = circular_views(2, 300.0, 450.0, 40, 40, 2.0, 2.0)  # outer pixels miss the volume
    got = host(pmf.conebeam_project(grid, Detector(40, 40, 1.0), views(vw), dev(vol), shared=True))
    ref = oracle.project(grid, 40, 40, 1.0, vw, vol)
    assert rel_l2(got, ref) <= TOL32
    assert np.all(got[ref == 0] == 0)


@pytest.mark.parametrize("shared", [False, True])
def test_backproject_matches_oracle_and_is_reproducible(shared):
    grid = Grid(20, 18, 14, 2.0, 2.0, 2.5)
    rng = np.random.default_rng(22)
    vw = circular_views(3, 400.0, 600.0, 29, 21, 1.8, 1.9, start=0.1)
    dY = rng.normal(size=(3, 21, 29)).astype(np.float32)
    det = Detector(29, 21, 1.0)
    got = pmf.conebeam_project_backward(grid, det, views(vw), dev(dY), shared=shared)
    again = pmf.conebeam_project_backward(grid, det, views(vw), dev(dY), shared=shared)
    assert torch.equal(got, again)
    ref = oracle.project_backward(grid, 29, 21, 1.0, vw, dY, shared=shared)
    assert rel_l2(host(got), ref) <= TOL32


def test_marchers_with_boxes_wider_than_32_voxels():
    """Samples one voxel apart, so a 48-sample chunk spans about 48 voxels
    along the rays and x-major tiles have boxes wider than 32 voxels: the plain
    staging and the adjoint hold them with rows 65 words apart (no chunk falls
    back), while the bulk copies, 44 voxels wide, gather those chunks from
    global memory instead.  Both staging forms still agree bit for bit and both
    directions match the oracle."""
    grid = Grid(64, 48, 24, 1.0, 1.0, 1.0)
    P, nu, nv = 4, 40, 24
    vw = circular_views(P, 300.0, 450.0, nu, nv, 0.2, 0.2, start=0.05)
    det = Detector(nu, nv, 1.0)
    vol = np.random.default_rng(81).random((P,) + grid.shape).astype(np.float32)
    vb = dev(vol).to(torch.bfloat16)
    pmf.device_counters(reset=True)
    y16 = pmf.conebeam_project(grid, det, views(vw), vb)  # plain staging
    assert pmf.device_counters(reset=True)["project_box_fallback"] == 0
    y32 = pmf.conebeam_project(grid, det, views(vw), vb.float())  # bulk copies
    assert pmf.device_counters(reset=True)["project_box_fallback"] > 0
    assert torch.equal(y32, y16)
    ref = oracle.project(grid, nu, nv, 1.0, vw, host(vb.float()))
    assert rel_l2(host(y32), ref) <= TOL32
    dY = np.random.default_rng(82).normal(size=(P, nv, nu)).astype(np.float32)
    got = pmf.conebeam_project_backward(grid, det, views(vw), dev(dY))
    assert pmf.device_counters(reset=True)["backproject_box_fallback"] == 0
    refb = oracle.project_backward(grid, nu, nv, 1.0, vw, dY)
    assert rel_l2(host(got), refb) <= TOL32


def test_loss_matches_oracle():
    rng = np.random.default_rng(5)
    a, b = rng.normal(size=(3, 17, 29)).astype(np.float32), rng.normal(size=(3, 17, 29)).astype(np.float32)
    for kind in (1, 2):
        loss, g = pmf.projection_loss(kind, dev(a), dev(b))
        lref, gref = oracle.loss(kind, a, b)
        assert float(loss.item()) == pytest.approx(lref, rel=1e-6)
        assert rel_l2(host(g), gref) <= 1e-6
        # arrays off the 16-byte grid (the kernel's scalar form)
        ua, ub = torch.zeros(a.size + 1, device="cuda"), torch.zeros(b.size + 1, device="cuda")
        ua[1:] = dev(a).reshape(-1)
        ub[1:] = dev(b).reshape(-1)
        loss_u, g_u = pmf.projection_loss(kind, ua[1:].reshape(a.shape), ub[1:].reshape(b.shape))
        assert float(loss_u.item()) == pytest.approx(lref, rel=1e-6)
        assert rel_l2(host(g_u), gref) <= 1e-6


def test_loss_at_the_paper_batch_size():
    """32 projections of 512x384 (the vectorised form over many grid-stride
    rounds) against a float64 sum."""
    rng = np.random.default_rng(6)
    a = rng.normal(size=(32, 384, 512)).astype(np.float32)
    b = rng.normal(size=(32, 384, 512)).astype(np.float32)
    for kind in (1, 2):
        loss, g = pmf.projection_loss(kind, dev(a), dev(b))
        lref, gref = oracle.loss(kind, a, b)
        assert float(loss.item()) == pytest.approx(lref, rel=1e-6)
        assert rel_l2(host(g), gref) <= 1e-6


# ------------------------------------------------------------- the chain

def _gpu_step(wl, meas, kind=2):
    g, det = wl.grid, wl.det
    ref = gset(wl.ref, wl.kappa)
    mbcs = [gset(m, wl.kappa) for m in wl.mbc]
    V = pmf.gs_voxelize(g, ref)[0]
    E = torch.stack([pmf.gs_voxelize(g, m) for m in mbcs])
    w = dev(wl.coeff)
    vt = views(wl.views)
    W = pmf.warp_combine(g, V, E, w)
    Y = pmf.conebeam_project(g, det, vt, W, shared=False)
    loss, dY = pmf.projection_loss(kind, Y, dev(meas))
    dW = pmf.conebeam_project_backward(g, det, vt, dY, shared=False)
    dV, dE, dw = pmf.warp_combine_backward(g, V, E, w, dW)
    gref = pmf.gs_voxelize_backward(g, ref, dV.reshape(1, *g.shape))
    gmbc = [pmf.gs_voxelize_backward(g, m, dE[l]) for l, m in enumerate(mbcs)]
    return loss, Y, dict(coeff=dw, ref=gref, mbc=gmbc, dV=dV, dE=dE, dW=dW)


@pytest.mark.parametrize("kind", [2, 1])
def test_full_chain_forward_and_gradients_match_oracle(kind):
    wl = fd_subproblem()
    meas = wl.measured
    loss, Y, grads = _gpu_step(wl, meas, kind)
    lref, gref, fref = oracle_chain.step(wl, meas, kind=kind)
    assert rel_l2(host(Y), fref["Y"]) <= TOL32
    assert float(loss.item()) == pytest.approx(lref, rel=1e-5)
    assert rel_l2(host(grads["coeff"]), gref["coeff"]) <= 1e-3
    for i in range(4):
        assert rel_l2(host(grads["ref"][i]), gref["ref"][i]) <= 1e-3
        for l in range(3):
            assert rel_l2(host(grads["mbc"][l][i]), gref["mbc"][l][i]) <= 1e-3


def test_small_workload_chain_forward_matches_oracle():
    wl = small_workload()
    loss, Y, _ = _gpu_step(wl, wl.measured)
    f = oracle_chain.forward(wl)
    assert rel_l2(host(Y), f["Y"]) <= TOL32


def test_projector_box_fallback_paths_match_oracle():
    """Pixels far larger than voxels make each chunk's voxel box exceed shared
    memory, forcing the global-memory paths of both projector and adjoint."""
    grid = Grid(40, 40, 40, 0.5, 0.5, 0.5)
    rng = np.random.default_rng(31)
    vol = rng.random(grid.shape).astype(np.float32)
    vw = circular_views(2, 60.0, 90.0, 18, 17, 12.0, 12.0, start=0.3)
    det = Detector(18, 17, 0.25)
    got = host(pmf.conebeam_project(grid, det, views(vw), dev(vol), shared=True))
    ref = oracle.project(grid, 18, 17, 0.25, vw, vol)
    assert rel_l2(got, ref) <= TOL32
    dY = rng.normal(size=(2, 17, 18)).astype(np.float32)
    gb = host(pmf.conebeam_project_backward(grid, det, views(vw), dev(dY), shared=True))
    assert rel_l2(gb, oracle.project_backward(grid, 18, 17, 0.25, vw, dY, shared=True)) <= TOL32


def test_projector_source_inside_volume():
    """Samples start at m = 0 when the source sits inside the padded volume."""
    grid = Grid(24, 24, 16, 2.0, 2.0, 2.0)
    vol = np.random.default_rng(32).random(grid.shape).astype(np.float32)
    vw = circular_views(3, 10.0, 60.0, 20, 14, 3.0, 3.0, start=0.2)
    det = Detector(20, 14, 1.0)
    got = host(pmf.conebeam_project(grid, det, views(vw), dev(vol), shared=True))
    assert rel_l2(got, oracle.project(grid, 20, 14, 1.0, vw, vol)) <= TOL32
    dY = np.random.default_rng(33).normal(size=(3, 14, 20)).astype(np.float32)
    gb = host(pmf.conebeam_project_backward(grid, det, views(vw), dev(dY), shared=True))
    assert rel_l2(gb, oracle.project_backward(grid, 20, 14, 1.0, vw, dY, shared=True)) <= TOL32


@pytest.mark.parametrize("L,std", [(3, 6.0), (1, 1.0), (4, 3.0)])
def test_fused_warp_tiles_with_large_displacements(L, std):
    """Ragged tiles (8x8x4 forward, 8x16x4 adjoint) and displacements well past the 4-voxel shared-memory
    halo (std 6 mm at 2 mm voxels): both the box and the direct scatter paths."""
    grid = Grid(37, 9, 7, 2.0, 2.0, 2.0)
    rng = np.random.default_rng(40 + L)
    V = rng.random(grid.shape).astype(np.float32)
    E = rng.normal(0, std, (L, 3) + grid.shape).astype(np.float32)
    w = rng.uniform(-1, 1, (5, L, 3)).astype(np.float32)
    dW = rng.normal(size=(5,) + grid.shape).astype(np.float32)
    D = oracle.combine(E, w)
    assert rel_l2(host(pmf.warp_combine(grid, dev(V), dev(E), dev(w))), oracle.warp(grid, V, D)) <= TOL32
    dV_ref, dD_ref = oracle.warp_backward(grid, V, D, dW)
    dE_ref, dw_ref = oracle.combine_backward(E, w, dD_ref)
    dV, dE, dw = pmf.warp_combine_backward(grid, dev(V), dev(E), dev(w), dev(dW))
    assert rel_l2(host(dV), dV_ref) <= TOL32
    assert rel_l2(host(dE), dE_ref) <= 1e-4
    assert rel_l2(host(dw), dw_ref) <= 1e-4


def test_voxelize_backward_unsplit_many_gaussians():
    """Enough Gaussians that each is handled by a single warp (no slab split)."""
    grid = Grid(40, 36, 30, 2.0, 2.0, 2.0)
    gs = _rand_gaussians(55, grid, 24000, 0.5, 2.0, 1)
    d_out = np.random.default_rng(56).normal(size=(1,) + grid.shape).astype(np.float32)
    got = pmf.gs_voxelize_backward(grid, gset(gs, 3.0), dev(d_out))
    ref = oracle.voxelize_backward(grid, gs.mean, gs.scale, gs.quat, gs.value, d_out, 3.0)
    for name, g_, r_ in zip(("mean", "scale", "quat", "value"), got, ref):
        assert rel_l2(host(g_), r_) <= 1e-4, name


@pytest.mark.parametrize("dt", [torch.float32, torch.bfloat16, torch.float16])
@pytest.mark.parametrize("n,L,P", [((8, 4, 3), 1, 1), ((8, 4, 3), 3, 2), ((7, 5, 3), 2, 1), ((7, 5, 3), 4, 5),
                                   ((33, 9, 5), 3, 4), ((12, 5, 4), 5, 3), ((12, 5, 4), 4, 9)])
def test_unfused_calls_at_run_and_tile_edges(n, L, P, dt):
    """mbc_combine, warp_volume and their adjoints where the four-voxel runs end
    (N a multiple of four or odd), past the 32 x 8 x 2 warp tile and the 8 x 16 x 4
    adjoint tile, for one view, a full group of four, a group and a rest, and
    more than four levels; displacements of up to a few voxels, some beyond the
    adjoint's 4-voxel halo.  fp32 sums: 1e-5 relative (reduced inputs are
    compared from the stored values, a reduced DVF to its half-ulp)."""
    grid = Grid(*n, 2.0, 2.0, 2.0)
    V, E, w = _mbc_and_ref(grid, 300 + L, L=L, P=P)
    Vd, Ed = dev(V).to(dt), dev(3.0 * E).to(dt)
    Vq, Eq = host(Vd), host(Ed)
    eps = {torch.float32: 1e-6, torch.bfloat16: 2.0 ** -8, torch.float16: 2.0 ** -11}[dt]
    D = pmf.mbc_combine(grid, Ed, dev(w))
    assert rel_l2(host(D), oracle.combine(Eq, w)) <= eps
    Dq = host(D)
    W = pmf.warp_volume(grid, Vd, D)
    assert rel_l2(host(W), oracle.warp(grid, Vq, Dq)) <= (TOL32 if dt == torch.float32 else eps)
    rng = np.random.default_rng(310 + P)
    dW = rng.normal(size=(P,) + grid.shape).astype(np.float32)
    dV, dD = pmf.warp_volume_backward(grid, Vd, D, dev(dW))
    dV_ref, dD_ref = oracle.warp_backward(grid, Vq, Dq, dW)
    assert rel_l2(host(dV), dV_ref) <= TOL32
    assert rel_l2(host(dD), dD_ref) <= 1e-4
    dV2, none = pmf.warp_volume_backward(grid, Vd, D, dev(dW), need_dvf=False)
    assert none is None and torch.equal(dV, dV2)
    g = rng.normal(size=(P, 3) + grid.shape).astype(np.float32)
    dE, dw = pmf.mbc_combine_backward(grid, Ed, dev(w), dev(g))
    dE_ref, dw_ref = oracle.combine_backward(Eq, w, g)
    assert rel_l2(host(dE), dE_ref) <= 1e-6
    assert rel_l2(host(dw), dw_ref) <= 1e-5
    base = (dE.clone(), dw.clone())
    pmf.mbc_combine_backward(grid, Ed, dev(w), dev(g), accumulate=True, grads=base)
    assert rel_l2(host(base[0]), 2.0 * dE_ref) <= 1e-6 and rel_l2(host(base[1]), 2.0 * dw_ref) <= 1e-5


@pytest.mark.parametrize("C", [1, 3])
@pytest.mark.parametrize("n,G,scale", [((37, 5, 3), 7, (0.4, 1.5)), ((150, 40, 30), 3, (8.0, 30.0))])
def test_voxelize_backward_row_plans(n, G, scale, C):
    """The adjoint numbers the blocks of 64 box rows at a time and lists 512 of
    them: a few rows, and rows as long as the grid (several listings per plan);
    against the oracle within the gradient bounds used above."""
    grid = Grid(*n, 2.0, 2.0, 2.0)
    gs = _rand_gaussians(400 + G, grid, G, scale[0] * 2.0, scale[1] * 2.0, C)
    d = np.random.default_rng(401 + G).normal(size=(C,) + grid.shape).astype(np.float32)
    got = pmf.gs_voxelize_backward(grid, gset(gs, 3.0), dev(d))
    ref = oracle.voxelize_backward(grid, gs.mean, gs.scale, gs.quat, gs.value, d, 3.0)
    for x, r in zip(got, ref):
        assert rel_l2(host(x), np.asarray(r).reshape(tuple(x.shape))) <= 1e-4


@pytest.mark.parametrize("C", [1, 3])
@pytest.mark.parametrize("accumulate", [False, True])
def test_voxelize_backward_of_a_crop(C, accumulate):
    """More Gaussians than the slabs' limit on a grid of fewer than four voxels
    per Gaussian takes eight Gaussians per warp: those outside the grid get zero
    (or nothing added), a sample of the others matches the oracle."""
    grid = Grid(17, 16, 15, 2.0, 2.0, 2.0)
    n = 20011  # above the slab limit of 152 * 64 * 4 / 2 warps, not a multiple of eight
    gs = _rand_gaussians(430, grid, n, 1.0, 4.0, C)
    gs.mean[::3] += np.float32(400.0)  # outside
    g = gset(gs, 3.0)
    d = dev(np.random.default_rng(431).normal(size=(C,) + grid.shape))
    base = [torch.full(s, 0.25, device="cuda") for s in ((n, 3), (n, 3), (n, 4), (n, C))]
    got = pmf.gs_voxelize_backward(grid, g, d, grads=tuple(base) if accumulate else None, accumulate=accumulate)
    for x in got:
        assert torch.all(x[::3] == (0.25 if accumulate else 0.0))
    sel = np.arange(1, n, 1500)
    ref = oracle.voxelize_backward(grid, gs.mean[sel], gs.scale[sel], gs.quat[sel], gs.value[sel], host(d), 3.0)
    for x, r in zip(got, ref):
        assert rel_l2(host(x)[sel] - (0.25 if accumulate else 0.0), np.asarray(r).reshape(len(sel), -1)) <= 1e-4


@pytest.mark.parametrize("G", [0, 1, 40])
def test_voxelize_without_workspace_takes_the_pair_bound(G):
    """A small call without a workspace allocates the list's bound, n x tiles,
    instead of counting: the same bits as with the exact count, whose value the
    bound covers."""
    grid = Grid(21, 17, 9, 2.0, 2.0, 2.0)
    gs = gset(_rand_gaussians(440, grid, max(G, 1), 1.0, 5.0, 3), 3.0)
    if G == 0:
        gs = pmf.Gaussians(gs.mean[:0], gs.scale[:0], gs.quat[:0], gs.value[:0], 3.0)
    exact = pmf.gs_voxelize_count(grid, gs)
    assert exact <= pmf.ops._pair_capacity(pmf.ops._grid(grid), gs) == G * 3 * 3 * 2
    assert torch.equal(pmf.gs_voxelize(grid, gs), pmf.gs_voxelize(grid, gs, pair_capacity=exact))


def test_voxelize_backward_on_a_grid_of_2_31_rows():
    """A grid one voxel wide whose last rows have an index past 2^31 (8.6 GB of
    upstream gradient): a Gaussian at that corner gets the gradient of the same
    Gaussian on a 41 x 41 patch with the same voxel centres (both axes odd, 1 mm
    voxels: every centre and difference is exact), within the bound used above."""
    n, m = 46401, 41
    grid, patch = Grid(1, n, n, 1.0, 1.0, 1.0), Grid(1, m, m, 1.0, 1.0, 1.0)
    assert (n - m) * n >= 2 ** 31
    d = np.random.default_rng(450).normal(size=(1, m, m, 1)).astype(np.float32)
    d_big = torch.zeros((1, n, n, 1), dtype=torch.float32, device="cuda")
    d_big[:, n - m:, n - m:] = dev(d)
    gs = gaussian_set(np.random.default_rng(451), patch, 1, 2.0, 3.0, channels=1)
    gs.mean[0] = (0.0, 0.25, -0.5)
    centre = (n - m) // 2  # the patch's centre voxel in the grid, mm from its own centre
    big = gset(gs, 3.0)
    big.mean[0, 1:] += float(centre)
    got = pmf.gs_voxelize_backward(grid, big, d_big)
    ref = oracle.voxelize_backward(patch, gs.mean, gs.scale, gs.quat, gs.value, d, 3.0)
    for x, r in zip(got, ref):
        assert rel_l2(host(x), np.asarray(r).reshape(tuple(x.shape))) <= 1e-4


@pytest.mark.parametrize("n,P", [((16, 9, 5), 2), ((32, 17, 9), 2), ((97, 9, 5), 1), ((33, 33, 33), 13),
                                 ((47, 33, 17), 21), ((32, 33, 33), 18)])
def test_unfused_warp_tile_shapes(n, P):
    """warp_volume and its adjoint on each tile: 32, 16 and 8 voxels wide (rows
    that fill less of the wider ones), one plane per lane (few blocks) and two;
    fp32 against the oracle within the bounds used above."""
    grid = Grid(*n, 2.0, 2.0, 2.0)
    rng = np.random.default_rng(460 + P)
    V = rng.random(grid.shape).astype(np.float32)
    D = (4.0 * rng.normal(size=(P, 3) + grid.shape)).astype(np.float32)
    dW = rng.normal(size=(P,) + grid.shape).astype(np.float32)
    assert rel_l2(host(pmf.warp_volume(grid, dev(V), dev(D))), oracle.warp(grid, V, D)) <= TOL32
    dV, dD = pmf.warp_volume_backward(grid, dev(V), dev(D), dev(dW))
    dV_ref, dD_ref = oracle.warp_backward(grid, V, D, dW)
    assert rel_l2(host(dV), dV_ref) <= TOL32
    assert rel_l2(host(dD), dD_ref) <= 1e-4


@pytest.mark.parametrize("tile", [None, (16, 8, 4)])
@pytest.mark.parametrize("extra", [0, 1, 63])
def test_voxelize_list_of_the_exact_count_lists_every_tile(tile, extra):
    """A list with room for the counted pairs, whatever the count's place in the
    workspace's 256-byte steps, holds them all: no tile scans every Gaussian (the
    last one did), and the volume is the same."""
    grid = Grid(30, 22, 13, 2.0, 2.0, 2.0)
    pmf.device_counters(reset=True)
    for n in (50, 57, 64, 71):
        gs = gset(_rand_gaussians(470 + n, grid, n, 0.7, 3.0, 1), 3.0)
        exact = pmf.gs_voxelize_count(grid, gs, tile)
        got = pmf.gs_voxelize(grid, gs, pair_capacity=exact + extra, tile=tile)
        assert torch.equal(got, pmf.gs_voxelize(grid, gs, tile=tile))
    assert pmf.device_counters()["voxelize_list_overflow"] == 0


@pytest.mark.parametrize("dt", [torch.float32, torch.bfloat16, torch.float16])
@pytest.mark.parametrize("n", [(41, 40, 39), (3, 2, 1)])
def test_project_gathered_chunks(n, dt):
    """Chunks whose box is too large to stage gather in pairs, from volumes with no
    16-byte rows: interior pairs, pairs across the volume's faces (every pair of
    the thin volume) and odd rests, against the oracle on the stored values."""
    grid = Grid(*n, 0.5, 0.5, 0.5)
    vw = circular_views(3, 60.0, 90.0, 18, 17, 12.0, 12.0, start=0.3)
    det = Detector(18, 17, 0.25)
    vol = dev(np.random.default_rng(490).random(grid.shape)).to(dt)
    pmf.device_counters(reset=True)
    got = pmf.conebeam_project(grid, det, views(vw), vol, shared=True)
    if n[0] > 3:
        assert pmf.device_counters(reset=True)["project_box_fallback"] > 0
    ref = oracle.project(grid, 18, 17, 0.25, vw, host(vol))
    assert rel_l2(host(got), ref) <= TOL32


@pytest.mark.parametrize("C,accumulate", [(1, False), (2, True), (3, False), (3, True), (4, False)])
@pytest.mark.parametrize("n,G,listed", [((17, 16, 15), 29184, True), ((17, 16, 15), 30011, True),
                                        ((17, 16, 15), 29183, False), ((53, 47, 41), 20011, False)])
def test_voxelize_backward_listed_and_warp_each(n, G, listed, C, accumulate):
    """The adjoint of a set too large to split: listed where there are fewer than
    four voxels and enough Gaussians, else a warp each, also on a volume of more
    voxels; about a third of the Gaussians outside get zero (or nothing added), a
    sample of the others at every place of a warp, the last ones among them,
    match the oracle within the bound used above."""
    grid = Grid(*n, 2.0, 2.0, 2.0)
    assert (4 * G > n[0] * n[1] * n[2]) == (n[0] < 50)
    assert (pmf.ops.gs_voxelize_backward_workspace(grid, G, C) > 0) == listed
    gs = _rand_gaussians(480, grid, G, 1.0, 4.0, C)
    gs.mean[::3] += np.float32(400.0)  # outside
    d = dev(np.random.default_rng(481).normal(size=(C,) + grid.shape))
    base = tuple(torch.full((G, k), 0.25, device="cuda") for k in (3, 3, 4, C)) if accumulate else None
    got = pmf.gs_voxelize_backward(grid, gset(gs, 3.0), d, grads=base, accumulate=accumulate)
    zero = 0.25 if accumulate else 0.0
    for x in got:
        assert torch.all(x[::3] == zero)
    sel = np.unique(np.concatenate([np.arange(0, G, 1499), np.arange(G - 8, G)]))
    sel = sel[sel % 3 != 0]
    ref = oracle.voxelize_backward(grid, gs.mean[sel], gs.scale[sel], gs.quat[sel], gs.value[sel], host(d), 3.0)
    for x, r in zip(got, ref):
        assert rel_l2(host(x)[sel] - zero, np.asarray(r).reshape(len(sel), -1)) <= 1e-4


def test_voxelize_backward_list_of_none():
    """A listed set with no Gaussian in the grid: zeros, or nothing added."""
    grid, G = Grid(9, 8, 7, 2.0, 2.0, 2.0), 30000
    gs = _rand_gaussians(482, grid, G, 1.0, 4.0, 1)
    gs.mean[:] += np.float32(400.0)
    d = torch.ones((1,) + grid.shape, device="cuda")
    assert all(float(x.abs().max()) == 0.0 for x in pmf.gs_voxelize_backward(grid, gset(gs, 3.0), d))


@pytest.mark.parametrize("n", [(8, 8, 8), (9, 8, 7)])
def test_marchers_take_steps_beyond_their_float_cells(n):
    """Steps that are infinite in voxels along x (a voxel of 1.2e-38 mm) or tens of
    thousands of voxels long leave the staged loops' float cells, so every such
    chunk goes through global memory, whose cells are checked integers: the calls
    return, the projections of the rays that cross are the NaN of a NaN position
    (or the oracle's value), and the next call is the usual one's."""
    vol = np.random.default_rng(491).random((2,) + n[::-1]).astype(np.float32)
    dY = torch.ones((2, 16, 16), device="cuda")
    vw = np.array([[0, -100, 1, 0, 100, 2, 1, 0, 0, 0, 0, 1.0], [3, -90, 0, -2, 110, 0, 1, 0, 0, 0, 0, 1.0]])
    thin, det = Grid(*n, 1.2e-38, 10.0, 10.0), Detector(16, 16, 5.0)
    pmf.device_counters(reset=True)
    for dt in (torch.float32, torch.bfloat16):
        Y = pmf.conebeam_project(thin, det, views(vw), dev(vol).to(dt))
        assert torch.all(torch.isnan(Y) | (Y == 0)) and torch.isnan(Y).any()
        Yb = pmf.conebeam_project_batched([(thin, det, views(vw), dev(vol).to(dt), False)])[0]
        assert torch.equal(torch.isnan(Yb), torch.isnan(Y))
    pmf.conebeam_project_backward(thin, det, views(vw), dY)
    c = pmf.device_counters(reset=True)
    assert c["project_box_fallback"] > 0 and c["backproject_box_fallback"] > 0 and c["timeout"] == 0
    # a step of 60,000 voxels from a source inside the volume: sample 0 and none other
    grid, far = Grid(*n, 2.0, 2.0, 2.0), Detector(16, 16, 120000.0)
    inside = circular_views(2, 1.0, 60.0, 16, 16, 3.0, 3.0, start=0.2)
    got = pmf.conebeam_project(grid, far, views(inside), dev(vol))
    ref = oracle.project(grid, 16, 16, 120000.0, inside, vol)
    assert rel_l2(host(got), ref) <= TOL32
    gb = pmf.conebeam_project_backward(grid, far, views(inside), dY)
    assert rel_l2(host(gb), oracle.project_backward(grid, 16, 16, 120000.0, inside, host(dY))) <= TOL32
    near = Detector(16, 16, 1.0)
    bt = pmf.conebeam_project_backward_batched([(grid, d, views(inside), dY, False) for d in (far, near)])
    assert torch.equal(bt[0], gb)
    refb = oracle.project_backward(grid, 16, 16, 1.0, inside, host(dY))
    assert rel_l2(host(bt[1]), refb) <= TOL32


def _flat_gaussians(rng, G, ratio, needles):
    """Rotated discs or needles of the axis ratio about a small grid's centre, half
    of them centred on voxel centres (which a flat one's ellipsoid else mostly
    misses)."""
    wide = np.exp(rng.uniform(np.log(3.0), np.log(8.0), G))
    thin = wide / ratio
    scale = np.stack([wide, thin if needles else wide * rng.uniform(0.6, 1.0, G), thin], 1).astype(np.float32)
    mean = rng.uniform(-16.0, 16.0, (G, 3))
    mean[::2] = 2.0 * np.round(mean[::2] / 2.0) + 1.0
    return mean.astype(np.float32), scale, rng.normal(size=(G, 4)).astype(np.float32), \
        rng.uniform(0.5, 1.0, (G, 1)).astype(np.float32)


@pytest.mark.parametrize("kappa", [3.0, float("inf")])
@pytest.mark.parametrize("needles", [False, True])
@pytest.mark.parametrize("ratio", [30.0, 100.0, 300.0])
def test_voxelize_keeps_flat_rotated_gaussians(ratio, needles, kappa):
    """The render drops sub-blocks that an ellipsoid cannot reach; a flat one's
    fp32 quadratic form loses digits to cancellation, which the drop must allow
    for.  With u = 2^-24, R's elements are good to 20 u (a normalised quaternion's
    products), so A's to sum_k (20 u (|R_ik| + |R_jk|) + 400 u^2 + 8 u |R_ik R_jk|) / s_k^2,
    and q is within that times |d_i d_j|, and 8 u more of its terms, of the exact
    one.  Every voxel lies between the sums with q that much larger and smaller,
    give or take the terms' 2^-21 rounding and fp32's; on every tile and without a
    list."""
    grid, G = Grid(20, 18, 16, 2.0, 2.0, 2.0), 60
    mean, scale, quat, value = _flat_gaussians(np.random.default_rng(int(ratio) + needles), G, ratio, needles)
    g = pmf.Gaussians(dev(mean), dev(scale), dev(quat), dev(value), kappa)
    got = pmf.gs_voxelize(grid, g)
    for tile in ((16, 8, 8), (8, 8, 4), (16, 8, 4)):
        assert torch.equal(got, pmf.gs_voxelize_tiled(grid, g, tile))
    assert torch.equal(got, pmf.gs_voxelize(grid, g, pair_capacity=0))
    u, ax = 2.0 ** -24, [(np.arange(n) + 0.5 - 0.5 * n) * 2.0 for n in (20, 18, 16)]
    X = np.stack(np.meshgrid(*ax, indexing="ij"), -1).transpose(2, 1, 0, 3)  # [nz, ny, nx, 3]
    lower, upper, k2 = 0.0, 0.0, kappa * kappa
    for m, s, q, v in zip(mean.astype(float), scale.astype(float), quat.astype(float), value[:, 0].astype(float)):
        w, x, y, z = q / np.linalg.norm(q)
        R = np.array([[1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y)],
                      [2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x)],
                      [2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)]])
        a = np.abs(R)
        M = (a / s ** 2) @ a.T
        E = 20 * u * ((a / s ** 2).sum(1)[:, None] + (a / s ** 2).sum(1)[None]) + 400 * u * u * (1 / s ** 2).sum() + 16 * u * M
        d = X - m
        qf = np.einsum("...i,ij,...j->...", d, (R / s ** 2) @ R.T, d)
        dq = np.einsum("...i,ij,...j->...", np.abs(d), E, np.abs(d))
        lower = lower + v * np.where(qf + dq <= k2, np.exp(-0.5 * (qf + dq)), 0.0)
        upper = upper + v * np.where(qf - dq <= k2, np.exp(-0.5 * np.maximum(qf - dq, 0.0)), 0.0)
    got, tol = host(got)[0], G * 2.0 ** -21 + 1e-6 * upper
    assert lower.sum() > 5.0 and np.all(got >= lower - tol) and np.all(got <= upper + tol)


@pytest.mark.parametrize("dt", [torch.float32, torch.bfloat16, torch.float16])
@pytest.mark.parametrize("L", [5, 6, 7, 8])
def test_combine_levels_above_four(L, dt):
    """mbc_combine at five to eight levels, in runs of four voxels and one by one
    (an odd voxel count): the sum in 32 bits over the stored vectors, rounded once."""
    tol = {torch.float32: TOL32, torch.bfloat16: 2.0**-8, torch.float16: 2.0**-11}[dt]
    for n, P in (((12, 6, 5), 3), ((11, 7, 5), 1), ((67, 66, 64), 2)):
        grid = Grid(*n, 2.0, 2.0, 2.0)
        rng = np.random.default_rng(490 + L)
        E = dev(rng.normal(size=(L, 3) + grid.shape).astype(np.float32)).to(dt)
        w = rng.normal(size=(P, L, 3)).astype(np.float32)
        got = pmf.mbc_combine(grid, E, dev(w))
        ref = np.einsum("plk,lkzyx->pkzyx", w.astype(np.float64), E.double().cpu().numpy())
        assert got.dtype == dt and rel_l2(host(got.float()), ref) <= tol


@pytest.mark.parametrize("nx,L,P", [(33, 1, 31), (33, 1, 32), (33, 2, 48), (33, 3, 64), (33, 4, 80), (33, 1, 95),
                                    (33, 1, 96), (33, 4, 128), (34, 1, 48), (34, 3, 111), (34, 3, 112)])
@pytest.mark.parametrize("dt", [torch.float32, torch.bfloat16])
def test_warp_combine_many_views_of_ragged_rows(nx, L, P, dt):
    """The fused forward at the view counts from which fewer CTAs run per SM (fp32
    rows not a multiple of four voxels): the same volumes as in calls of 16 views."""
    grid = Grid(nx, 130, 131, 2.0, 2.0, 2.0)
    V, E, w = _mbc_and_ref(grid, 500 + P, L=L, P=P)
    Vd, Ed, wd = dev(V).to(dt), dev(E).to(dt), dev(w)
    out = torch.full((P,) + grid.shape, float("nan"), device="cuda")
    got = pmf.warp_combine(grid, Vd, Ed, wd, out=out)
    for p in range(0, P, 16):
        part = torch.empty((min(16, P - p),) + grid.shape, device="cuda")
        assert torch.equal(got[p:p + 16], pmf.warp_combine(grid, Vd, Ed, wd[p:p + 16], out=part))
