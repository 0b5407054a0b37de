"""Previews by the number of rays of a launch: eight or four lanes per ray, or 8,
16 or 32 rays per warp, in launches of their own and in batches.  The image is
the same bit for bit, at the sizes where the choice changes and beside larger
previews in one batch, and the middle form agrees with the oracle."""
import numpy as np
import pytest

import vdi_synth as S
from helpers import check_with_alternatives, preview_alternatives, random_case

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


SIZES = [(250, 200), (251, 200), (500, 320), (533, 301), (500, 400), (501, 400), (640, 360), (600, 500), (601, 500),
         (1200, 1000), (1201, 1000)]


@pytest.mark.parametrize("w, h, ns, fmt, d_r", [(40, 24, 2, 1, 2), (67, 41, 5, 0, 4), (33, 65, 33, 1, 2)])
def test_preview_forms_agree(V, ctx, w, h, ns, fmt, d_r):
    case = random_case(w, h, ns, seed=w + 1)
    vdi = V.vdi_create(ctx, case.gpu_desc(V, fmt), case.vdi.rgba, case.vdi.depth, case.vdi.counts)
    try:
        for W, H in SIZES:
            cn = S.orbit_camera(case.bmin, case.bmax, W / H, az_deg=30, el_deg=15)
            cam = V.camera(cn.view, cn.proj)
            one, alone, beside = (torch.zeros((H, W, 4), device="cuda") for _ in range(3))
            big = torch.zeros((500, 601, 4), device="cuda")
            V.vdi_render(vdi, cam, W, H, 1, d_r, one)
            V.vdi_render_batch(ctx, [V.request(vdi, cam, W, H, 1, d_r, alone)])
            V.vdi_render_batch(ctx, [V.request(vdi, cam, W, H, 1, d_r, beside), V.request(vdi, cam, 601, 500, 1, d_r, big)])
            assert one[..., 3].max() > 0 and torch.equal(one, alone) and torch.equal(one, beside), (W, H)
    finally:
        V.vdi_destroy(vdi)


@pytest.mark.parametrize("W,H", [(75, 53), (441, 250), (533, 301)])
def test_preview_forms_match_the_oracle(V, ctx, orc, W, H):
    T, nz = 8, 10
    case = random_case(64, 48, 6, seed=21, u=0.15, alpha_range=(0.05, 0.6))
    sc = case.oracle_scene(orc)
    grid = orc.grid_counts(sc, T, nz)
    vdi = V.vdi_create(ctx, case.gpu_desc(V, 0, T, nz), case.vdi.rgba, case.vdi.depth, case.vdi.counts)
    try:
        cn = S.orbit_camera(case.bmin, case.bmax, W / H, az_deg=20.0, el_deg=10.0, zoom=1.1)
        cam = V.camera(cn.view, cn.proj)
        one, alone = (torch.zeros((H, W, 4), device="cuda") for _ in range(2))
        V.vdi_render(vdi, cam, W, H, 1, 2, one)
        V.vdi_render_batch(ctx, [V.request(vdi, cam, W, H, 1, 2, alone)])
        torch.cuda.synchronize()
    finally:
        V.vdi_destroy(vdi)
    ref, fl = orc.render_preview(sc, cn.view, cn.proj, W, H, 2, T, nz, grid=grid)
    assert ref[:, 3].max() > 0.2
    alts = preview_alternatives(orc, sc, cn, W, H, 2, T, nz, grid, np.nonzero(fl)[0])
    for got in (one, alone):
        frac, _ = check_with_alternatives(got.cpu().numpy(), ref, 0, fl, alts, what=f"preview {W}x{H}")
        assert frac < 0.2


def test_a_small_preview_in_a_batch_costs_like_one_alone(V, ctx):
    """A batch of one small preview (the serving loop's usual batch) against the same
    preview in a launch of its own, on the device: no more than 1.9 times as long (two
    launches and a tile queue for one launch); 2.8 times with 16 rays per warp."""
    n = 128
    vol = torch.from_numpy(S.value_noise_volume(n, seed=3, dtype=np.uint16)).cuda()
    bmin, bmax = np.zeros(3), np.ones(3)
    co = S.orbit_camera(bmin, bmax, 16 / 9, el_deg=20.0)
    vdi = V.vdi_generate(ctx, vol, bmin, bmax, S.tf_knots("sparse"), V.camera(co.view, co.proj), 640, 360, 20, 0.01, 1 / n,
                         1 / n, V.VDI_F16)
    try:
        W = H = 64
        cn = S.orbit_camera(bmin, bmax, 1.0, az_deg=30.0, el_deg=20.0)
        cam = V.camera(cn.view, cn.proj)
        out = torch.zeros((H, W, 4), device="cuda")
        req = [V.request(vdi, cam, W, H, 1, 2, out)]

        def us(fn):
            best = 1e9
            for _ in range(6):
                a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
                torch.cuda._sleep(3000000)
                a.record()
                for _ in range(20):
                    fn()
                b.record()
                torch.cuda.synchronize()
                best = min(best, a.elapsed_time(b) / 20 * 1e3)
            return best

        one = us(lambda: V.vdi_render(vdi, cam, W, H, 1, 2, out))
        batch = us(lambda: V.vdi_render_batch(ctx, req))
        assert batch < 1.9 * one
    finally:
        V.vdi_destroy(vdi)
