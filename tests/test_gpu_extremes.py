"""Inputs at the edges of what the calls accept: pixels that overflow FP32
variances, infinite and NaN pixels, sums whose terms differ by many orders of
magnitude, eyes so far away that FP32 positions miss the box."""
import math
import time

import numpy as np
import pytest

from helpers import random_case

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def V():
    import paper_2206_08660_gb300 as V

    V.load()
    return V


@pytest.fixture(scope="module")
def ctx(V):
    c = V.vdi_ctx_create(0)
    yield c
    V.vdi_ctx_destroy(c)


@pytest.mark.parametrize("W,H", [(7, 7), (9, 12), (70, 45)])
@pytest.mark.parametrize("which", [0, 1, 2])
def test_ssim_where_a_variance_overflows(V, W, H, which):
    """Finite pixels of alternating sign whose sum of squares leaves FP32 while
    the means and the covariance do not: SSIM is about 0 there, not NaN."""
    from oracle import quality as Q

    rng = np.random.default_rng(W)
    sign = 1.0 - 2.0 * (np.add.outer(np.arange(H), np.arange(W)) % 2)
    huge = np.repeat((3e19 * sign)[..., None], 4, axis=2).astype(np.float32)
    plain = rng.uniform(0, 1, (H, W, 4)).astype(np.float32)
    a, b = [(huge, plain), (plain, huge), (huge, 0.5 * huge)][which]
    ssim, _ = V.vdi_image_quality(torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda())
    if which < 2:
        assert abs(Q.ssim(a, b)) < 1e-6 and abs(ssim) < 2e-6
    else:  # the covariance overflows too: inf / inf
        assert math.isnan(ssim)


@pytest.mark.parametrize("fmt", [0, 1])
@pytest.mark.parametrize("at", [(0, 0), (3, 5), (18, 37), (44, 69)])
@pytest.mark.parametrize("pa, pb, psnr", [(float("nan"), 0.5, "inf"), (float("inf"), 0.5, "-inf"), (0.5, float("-inf"), "-inf"),
                                          (float("inf"), float("inf"), "inf")])
def test_quality_of_infinite_and_nan_pixels(V, fmt, at, pa, pb, psnr):
    """SSIM is NaN; PSNR is -inf at an infinite error and +inf where the error is
    NaN (the call's value for a mean squared error that is not above 0)."""
    W, H = 70, 45
    rng = np.random.default_rng(1)
    img = [rng.uniform(0, 1, (H, W, 4)).astype(np.float32) for _ in range(2)]
    for k, p in enumerate((pa, pb)):
        img[k][at[0], at[1], 1] = p
    dt = torch.float32 if fmt == 0 else torch.float16
    ssim, got = V.vdi_image_quality(*[torch.from_numpy(i).to(dt).cuda() for i in img], fmt)
    assert math.isnan(ssim)
    assert got == float(psnr)
    for k in range(2):  # the fourth channel is not measured
        img[k][at[0], at[1], 1] = 0.5
        img[k][at[0], at[1], 3] = (pa, pb)[k]
    ssim, got = V.vdi_image_quality(*[torch.from_numpy(i).to(dt).cuda() for i in img], fmt)
    assert math.isfinite(ssim) and math.isfinite(got)


@pytest.mark.parametrize("colours", [((0.3, 0.7), (0.0, 1.0), (0.0, 1000.0)), ((0.31, 0.77), (0.0, 30.7), (0.0, 777.7))])
def test_ssim_sums_in_fp64(V, colours):
    """Constant channels: every window of a channel has the same FP32 value, so
    the image's SSIM is their exact mean up to the rounding of 12 additions and a
    division in FP64 (16 half ulps), whatever the terms' magnitudes."""

    def ssim(H, ch):
        ab = np.asarray(ch, np.float32).T  # [2, 3]
        img = [np.ascontiguousarray(np.broadcast_to(np.append(c, 1).astype(np.float32), (H, 7, 4))) for c in ab]
        return V.vdi_image_quality(*[torch.from_numpy(i).cuda() for i in img])[0]

    w = [ssim(7, [c] * 3) for c in colours]  # one window per channel
    assert all(x == float(np.float32(x)) for x in w)
    exact = math.fsum(w * 4) / 12
    assert abs(ssim(10, colours) - exact) <= 16 * 2.0 ** -53 * exact


@pytest.mark.parametrize("W,H", [(7, 7), (8, 22), (33, 9), (320, 200), (1024, 48), (256, 256), (513, 129), (700, 300)])
def test_quality_by_image_size(V, W, H):
    """One window per thread in images of fewer than 128 blocks of 32 x 16
    windows, four in larger ones: the oracle's measures on both sides."""
    from oracle import quality as Q

    rng = np.random.default_rng(W + H)
    a = rng.uniform(0, 1, (H, W, 4)).astype(np.float32)
    b = np.clip(a + rng.normal(0, 0.05, a.shape), 0, 1).astype(np.float32)
    ssim, psnr = V.vdi_image_quality(torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda())
    assert abs(ssim - Q.ssim(a, b)) < 2e-6 and abs(psnr - Q.psnr(a, b)) < 1e-6


def far_camera(D):
    """An eye at (-D, 1/2, 1/2) looking along x at a box one unit across."""
    view = np.array([[0, 0, 1, -0.5], [0, 1, 0, -0.5], [-1, 0, 0, -D], [0, 0, 0, 1.0]])
    near, far = D / 2, 2 * D
    proj = np.zeros((4, 4))
    proj[0, 0] = proj[1, 1] = 4 * D
    proj[2, 2], proj[2, 3], proj[3, 2] = -(far + near) / (far - near), -2 * far * near / (far - near), -1.0
    return view, proj


@pytest.mark.parametrize("dtype", [np.uint8, np.uint16, np.float32])
@pytest.mark.parametrize("log_d", [41, 46, 30])
@pytest.mark.parametrize("axis", [0, 1])
def test_sampling_from_a_distant_eye(V, ctx, orc, dtype, log_d, axis):
    """FP32 positions are up to 2^23 units apart: they fall on either side of the
    box, up to 2^29 voxels away, and read its first and last voxels, as plain
    arithmetic does.  (A box half an ulp of the eye's distance away from the
    origin keeps an interval between its faces.)"""
    D = 2.0 ** log_d
    ulp = D * 2.0 ** -23
    dims = [1, 1, 1]
    dims[2 - axis] = 128  # along the view, or across it
    top = 1.0 if dtype == np.float32 else np.iinfo(dtype).max
    vol = np.zeros(dims, dtype)
    vol.reshape(-1)[:64] = top
    kn = np.array([[0, 0.1, 0.2, 0.9, 0.01], [1, 0.9, 0.3, 0.1, 0.02]], np.float32)
    bmin = np.array([max(ulp / 2 - 0.5, 0.0), 0, 0])
    bmax = bmin + [1, 1, 1]
    view, proj = far_camera(D)
    step = max(ulp / 2.0 ** 12, 1.0)
    args = (kn, view, proj, 6, 5)
    ref = orc.dvr(orc.Volume(vol, bmin, bmax), *args, step, step, fp32=True)
    out = torch.zeros((5, 6, 4), device="cuda")
    V.vdi_dvr(ctx, torch.from_numpy(vol).cuda(), bmin, bmax, kn, V.camera(view, proj), 6, 5, step, step, out)
    assert ref[:, 3].min() > 0.5
    assert np.abs(out.cpu().numpy().reshape(-1, 4) - ref).max() < 1e-5


@pytest.mark.parametrize("offset", [1, 2, 3, 4])
def test_create_with_unaligned_device_counts(V, ctx, offset):
    """Device counts at any byte address, as a copy takes them."""
    case = random_case(37, 21, 5, seed=2)
    a = case.vdi
    rgba, depth = torch.from_numpy(a.rgba).cuda(), torch.from_numpy(a.depth).cuda()
    raw = torch.zeros(4 * a.counts.size + 8, dtype=torch.uint8, device="cuda")
    counts = raw[offset:offset + 4 * a.counts.size]
    counts.copy_(torch.from_numpy(np.ascontiguousarray(a.counts, np.int32).view(np.uint8).reshape(-1)))
    assert counts.data_ptr() % 4 == offset % 4
    vdi = V.vdi_create(ctx, case.gpu_desc(V, V.VDI_F32), rgba, depth, counts)
    try:
        assert np.array_equal(V.vdi_download(vdi, a.w, a.h, a.ns)[2], a.counts)
    finally:
        V.vdi_destroy(vdi)


def test_large_grid_cells_keep_the_gpu_busy(V, ctx):
    """Building a VDI with 64 or 256 lists per cell edge, against the default of 8: 1.1
    and 5.5 times as long on GB300 (a cell is one block's work, and 1920 x 1080
    lists have 40 cells of 256); 4.7 and 50 times with eight such cells to a block."""
    w, h, ns = 1920, 1080, 20
    edge = torch.linspace(-0.5, 0.9, 2 * ns, device="cuda").view(1, 1, ns, 2)
    depth = edge.expand(h, w, ns, 2).contiguous()
    rgba = torch.tensor([0.1, 0.2, 0.1, 0.3], device="cuda").expand(h, w, ns, 4).contiguous()
    n = torch.where(torch.rand(h, w, device="cuda") < 0.25, ns, 0).int()
    case = random_case(4, 4, 1, seed=1)
    best = {}
    for T in (8, 64, 256):
        d = V.desc(w, h, ns, case.cam_o.view, case.cam_o.proj, case.bmin, case.bmax, case.u, V.VDI_F16, grid_tile=T)
        for _ in range(4):
            torch.cuda.synchronize()
            t = time.perf_counter()
            vdi = V.vdi_create(ctx, d, rgba, depth, n)
            torch.cuda.synchronize()
            best[T] = min(best.get(T, 1e9), time.perf_counter() - t)
            V.vdi_destroy(vdi)
    assert best[64] < 2.5 * best[8] and best[256] < 20 * best[8]
