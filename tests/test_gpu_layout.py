"""The arrays beside a VDI's slots: count grid and block ranges over cell sizes
and shapes at the edges of the kernel's blocks (eight cells wide, 512 lists at a
time), supersegments that start, end or lie on slab edges, and empty lists."""
import numpy as np
import pytest

from helpers import random_case
import vdi_synth as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def V():
    import paper_2206_08660_gb300 as V

    V.load()
    return V


@pytest.fixture(scope="module")
def orc():
    import oracle

    oracle.build()
    return oracle


@pytest.fixture(scope="module")
def ctx(V):
    c = V.vdi_ctx_create(0)
    yield c
    V.vdi_ctx_destroy(c)


@pytest.mark.parametrize("w, h, ns, T, nz, device", [
    (1, 1, 1, 8, 1, False), (65, 9, 5, 8, 20, True), (64, 8, 16, 8, 64, False), (33, 17, 17, 8, 20, True),
    (40, 13, 3, 3, 7, False), (70, 30, 4, 12, 5, True), (95, 41, 6, 64, 20, False), (130, 20, 2, 256, 20, True),
    (9, 5, 33, 1, 20, True)])
def test_grid_and_block_ranges(V, ctx, orc, w, h, ns, T, nz, device):
    case = random_case(w, h, ns, seed=w + ns)
    vdi_a = case.vdi
    e = orc.grid_edges(case.oracle_scene(orc), nz)
    rng = np.random.default_rng(1)
    for iy, ix in zip(*np.nonzero(vdi_a.counts > 0)):  # a supersegment's face moved onto the slab edge inside it
        j = rng.integers(vdi_a.counts[iy, ix])
        f, b = vdi_a.depth[iy, ix, j]
        inside = e[(e >= f) & (e <= b)]
        if len(inside):
            vdi_a.depth[iy, ix, j, rng.integers(2)] = inside[0]
            if rng.random() < 0.3:
                vdi_a.depth[iy, ix, j] = inside[0]
    arrays = (vdi_a.rgba, vdi_a.depth, vdi_a.counts)
    if device:
        arrays = [torch.as_tensor(a, device="cuda") for a in arrays]
    d = V.desc(w, h, ns, case.cam_o.view, case.cam_o.proj, case.bmin, case.bmax, case.u, V.VDI_F32, grid_tile=T, grid_nz=nz)
    for counts in (arrays[2], None):  # given, or counted from the finite depths
        vdi = V.vdi_create(ctx, d, arrays[0], arrays[1], counts)
        try:
            rgba, depth, n, grid = V.vdi_download(vdi, w, h, ns)
            assert np.array_equal(grid, orc.grid_counts(case.oracle_scene(orc), T, nz))
            assert np.array_equal(n, vdi_a.counts)
            dead = np.arange(ns)[None, None, :] >= vdi_a.counts[..., None]
            assert np.array_equal(depth[~dead], vdi_a.depth[~dead]) and np.all(np.isposinf(depth[dead]))
            W, H = 61, 37
            cn = S.orbit_camera(case.bmin, case.bmax, W / H, az_deg=25, el_deg=10)
            img = [torch.zeros((H, W, 4), device="cuda") for _ in range(2)]
            for out, blocks in zip(img, (False, True)):
                V.vdi_render_ex(vdi, V.camera(cn.view, cn.proj), W, H, 1, 1, out, blocks=blocks)
            assert torch.equal(img[0], img[1])
        finally:
            V.vdi_destroy(vdi)


@pytest.mark.parametrize("w, h, ns, fmt", [(1, 1, 1, 0), (40, 24, 2, 1), (67, 41, 3, 0), (33, 65, 20, 1), (16, 9, 64, 0)])
def test_walk_equals_the_searching_walk(V, ctx, w, h, ns, fmt):
    """The exact frame's walk (seed pair, neighbouring pair, then a search; 16 or
    32 rays per warp by launch size) against the walk that searches every list
    from scratch: the same image, bit for bit, for depth rising and falling
    along the rays, boxes that leave the frustum, and images of one tile, of few
    and of many."""
    case = random_case(w, h, ns, seed=w * ns)
    vdi = V.vdi_create(ctx, case.gpu_desc(V, fmt), case.vdi.rgba, case.vdi.depth, case.vdi.counts)
    try:
        for W, H, az, el, zoom in ((1, 1, 20, 0, 1.0), (31, 9, 2, 15, 1.0), (200, 150, 35, -20, 1.0), (640, 400, 100, 30, 1.5),
                                   (500, 333, 178, 10, 1.0)):
            cn = S.orbit_camera(case.bmin, case.bmax, W / H, az_deg=az, el_deg=el, zoom=zoom)
            img = [torch.zeros((H, W, 4), device="cuda") for _ in range(2)]
            for out, search in zip(img, (V.VDI_SEARCH_ALG2, V.VDI_SEARCH_BINARY)):
                V.vdi_render_ex(vdi, V.camera(cn.view, cn.proj), W, H, 1, 1, out, search=search)
            assert torch.equal(img[0], img[1]), (W, H, az)
    finally:
        V.vdi_destroy(vdi)


@pytest.mark.parametrize("w, h, ns, fmt", [(40, 24, 2, 1), (67, 41, 5, 0), (33, 65, 33, 1)])
def test_preview_rays_per_warp(V, ctx, w, h, ns, fmt):
    """Previews at the sizes where the rays per warp change (4, 8 or 16 in a launch
    of its own, 16 in a batch): the same image, bit for bit."""
    case = random_case(w, h, ns, seed=w)
    vdi = V.vdi_create(ctx, case.gpu_desc(V, fmt), case.vdi.rgba, case.vdi.depth, case.vdi.counts)
    try:
        for W, H in ((5, 3), (40, 30), (500, 300), (800, 600), (1601, 903)):
            cn = S.orbit_camera(case.bmin, case.bmax, W / H, az_deg=30, el_deg=15)
            cam = V.camera(cn.view, cn.proj)
            img = [torch.zeros((H, W, 4), device="cuda") for _ in range(2)]
            V.vdi_render(vdi, cam, W, H, 1, 2, img[0])
            V.vdi_render_batch(ctx, [V.request(vdi, cam, W, H, 1, 2, img[1])])
            assert img[0][..., 3].max() > 0 and torch.equal(img[0], img[1]), (W, H)
    finally:
        V.vdi_destroy(vdi)
