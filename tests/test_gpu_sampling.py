"""Volume sampling of vdi_generate and vdi_dvr: the fast forms (multiplications
with precomputed reciprocals, floor and conversion through the mantissa) and the
general one (plain divisions) take the same FP32 decisions as the oracle's IEEE
generation, over voxel types, ragged and one-voxel-thin volumes, boxes of other
extents than 1 and transfer functions of 2 to 16 knots."""
import numpy as np
import pytest

import vdi_synth as S

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


def make_volume(dtype, dims, seed):
    rng = np.random.default_rng(seed)
    k = rng.random((4, 4, 4))
    idx = [np.minimum((np.arange(n) * 4) // n, 3) for n in dims]
    v = k[np.ix_(*idx)] * 0.7 + 0.3 * rng.random(dims)
    if dtype == np.float32:
        return v.astype(np.float32)
    top = np.iinfo(dtype).max
    return np.rint(v * top).astype(dtype)


def make_knots(n, lowest):
    rng = np.random.default_rng(n)
    k = np.zeros((n, 5), np.float32)
    k[:, 0] = np.sort(rng.uniform(0.05, 0.95, n)).astype(np.float32)
    k[0, 0] = lowest
    k[:, 1:4] = rng.random((n, 3))
    k[:, 4] = rng.uniform(0.0, 0.2, n)
    k[0, 4] = 0.0
    return k


BOXES = {"unit": ([0, 0, 0], [1, 1, 1]), "ragged": ([-0.3, 0.1, 0.2], [0.9, 0.8, 1.35])}


@pytest.mark.parametrize("dtype", [np.uint8, np.uint16, np.float32])
@pytest.mark.parametrize("dims", [(32, 32, 32), (17, 29, 33), (1, 24, 40), (40, 3, 1)])
@pytest.mark.parametrize("box", list(BOXES))
@pytest.mark.parametrize("knots,lowest", [(2, 0.0), (4, 0.2), (5, 0.0), (16, 0.01), (4, 1e-30)])  # the last: general form
def test_generation_decisions_match_oracle(V, ctx, orc, dtype, dims, box, knots, lowest):
    w, h, ns, tau = 45, 27, 7, 0.01
    bmin, bmax = (np.asarray(b, np.float64) for b in BOXES[box])
    vol, kn = make_volume(dtype, dims, 3), make_knots(knots, lowest)
    u = float((bmax - bmin).max()) / 40
    cam = S.orbit_camera(bmin, bmax, w / h, az_deg=17, el_deg=20)
    args = (kn, cam.view, cam.proj, w, h, ns, tau, u, u)
    rgba, depth, counts = orc.generate(orc.Volume(vol, bmin, bmax), *args, fp32=True)
    g = V.vdi_generate(ctx, torch.from_numpy(vol).cuda(), bmin, bmax, kn, V.camera(cam.view, cam.proj), w, h, ns, tau, u,
                       u, V.VDI_F32)
    try:
        g_rgba, g_depth, g_counts, _ = V.vdi_download(g, w, h, ns)
    finally:
        V.vdi_destroy(g)
    assert counts.sum() > 0
    assert np.array_equal(g_counts, counts)
    valid = np.arange(ns)[None, None, :] < counts[:, :, None]
    assert np.array_equal(g_depth[valid].view(np.uint32), depth[valid].view(np.uint32))
    assert np.abs(g_rgba[valid] - rgba[valid]).max() < 2e-5  # as the existing generation tests


@pytest.mark.parametrize("dtype", [np.uint8, np.uint16, np.float32])
@pytest.mark.parametrize("form", ["recorded", "few rays", "empty", "general", "deep"])
def test_adaptive_forms_match_oracle(V, ctx, orc, dtype, form):
    """Algorithm 3 from recorded samples (whole and ragged tiles, rays without a
    sample), and its two other routes: general sampling, and rays of so many
    samples (14,000) that they are not recorded.  Gamma, counts and depths are
    the oracle's."""
    w, h = {"few rays": (3, 2), "deep": (16, 9)}.get(form, (45, 27))
    ns, steps = 7, 8200 if form == "deep" else 40
    bmin, bmax = np.zeros(3), np.ones(3)
    vol, kn = make_volume(dtype, (24, 20, 28), 5), make_knots(4, 1e-30 if form == "general" else 0.2)
    if form == "empty":
        vol[:] = 0
    if form == "deep":
        kn[:, 4] *= 0.01
    u = 1.0 / steps
    cam = S.orbit_camera(bmin, bmax, w / h, az_deg=30, el_deg=20)
    args = (kn, cam.view, cam.proj, w, h, ns, 0.0, u, u)
    rgba, depth, counts, tau = orc.generate(orc.Volume(vol, bmin, bmax), *args, fp32=True, adaptive=True, with_tau=True)
    t = torch.zeros((h, w), dtype=torch.float32, device="cuda")
    g = V.vdi_generate(ctx, torch.from_numpy(vol).cuda(), bmin, bmax, kn, V.camera(cam.view, cam.proj), w, h, ns, 0.0, u, u,
                       V.VDI_F32, adaptive=True, tau_out=t)
    try:
        g_rgba, g_depth, g_counts, _ = V.vdi_download(g, w, h, ns)
    finally:
        V.vdi_destroy(g)
    assert (counts.sum() == 0) == (form == "empty")
    assert np.array_equal(t.cpu().numpy(), tau.reshape(h, w))
    assert np.array_equal(g_counts, counts)
    valid = np.arange(ns)[None, None, :] < counts[:, :, None]
    assert np.array_equal(g_depth[valid].view(np.uint32), depth[valid].view(np.uint32))
