"""Device memory of adaptive generation: its scratch is bounded, given back with
the context, and counted by the server that generates; a budget without room for
it still generates the same VDI."""
import os
import subprocess
import sys

import numpy as np
import pytest

import vdi_synth as S

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

MEMORY = """
import numpy as np, torch
import vdi_synth as S
import paper_2206_08660_gb300 as V
n = 512
vol = torch.randint(0, 3, (n, n, n), dtype=torch.uint8, device="cuda")
cam = S.orbit_camera(np.zeros(3), np.ones(3), 16 / 9, el_deg=20.0)
kn = S.tf_knots("sparse")
def generate(ctx, **kw):
    V.vdi_destroy(V.vdi_generate(ctx, vol, np.zeros(3), np.ones(3), kn, V.camera(cam.view, cam.proj), 640, 360, 8, 0.01,
                                 0.5 / n, 1.0 / n, V.VDI_F16, **kw))
    torch.cuda.synchronize()
def free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]
ctx = V.vdi_ctx_create(0)
generate(ctx)  # the VDI's own memory, kept by the pool, and the kernels
a = free()
for _ in range(3):
    generate(ctx, adaptive=True)
b = free()
V.vdi_ctx_destroy(ctx)
print((a - b) >> 20, (a - free()) >> 20)
"""


def test_adaptive_scratch_is_bounded_and_given_back():
    """512^3 voxels at half-voxel steps: 840 MB of scratch for every warp the GPU
    holds; at most 512 MiB are taken and kept, and none after the context."""
    r = subprocess.run([sys.executable, "-c", MEMORY], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    kept, after = (int(x) for x in r.stdout.split())
    assert 64 < kept <= 512 + 64 and after <= 64, (kept, after)


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


@pytest.mark.parametrize("spare_mib", [2, 200, 4000])
def test_server_charges_adaptive_scratch(V, ctx, spare_mib):
    n, w, h, ns = 128, 320, 180, 12
    vol = torch.from_numpy(S.value_noise_volume(n, seed=4, dtype=np.uint16)).cuda()
    bmin, bmax = np.zeros(3), np.ones(3)
    co = S.orbit_camera(bmin, bmax, w / h, el_deg=20.0)
    kn, cam_o = S.tf_knots("sparse"), V.camera(co.view, co.proj)
    cn = S.orbit_camera(bmin, bmax, w / h, az_deg=15.0, el_deg=20.0)
    cam = V.camera(cn.view, cn.proj)
    ref = torch.zeros((h, w, 4), device="cuda")
    vdi = V.vdi_generate(ctx, vol, bmin, bmax, kn, cam_o, w, h, ns, 0.0, 1 / n, 1 / n, V.VDI_F32, adaptive=True)
    held = V.vdi_get_layout(vdi).total_bytes
    V.vdi_render(vdi, cam, w, h, 1, 1, ref)
    torch.cuda.synchronize()
    V.vdi_destroy(vdi)
    budget = held + (spare_mib << 20)
    srv = V.vdi_server_create(ctx, budget_bytes=budget, n_slots=1)
    try:
        side = torch.cuda.Stream()
        with torch.cuda.stream(side):
            torch.cuda._sleep(200_000_000)  # the generation waits behind it, in flight
        V.vdi_server_generate(srv, 0, vol, bmin, bmax, kn, cam_o, w, h, ns, 0.0, 1 / n, 1 / n, V.VDI_F32, stream=side,
                              adaptive=True)
        st = V.vdi_server_stats(srv)
        assert st.vdi_bytes == held
        if spare_mib == 2:  # no scratch that would help fits half of 2 MiB: sampled at every gamma
            assert st.bytes_in_use == 0
        else:
            assert (1 << 20) < st.bytes_in_use <= (spare_mib << 20) // 2 and st.bytes_in_use <= 512 << 20
        t = V.vdi_server_submit(srv, V.view_request(0, cam, w, h, out_fmt=V.VDI_F32))
        info = V.vdi_server_wait(srv, t, 30.0)
        assert info.status == 0
        out = torch.zeros_like(ref)
        V.vdi_server_read(srv, t, out)
        assert torch.equal(out, ref)
        V.vdi_server_release(srv, t)
        torch.cuda.synchronize()
        assert V.vdi_server_stats(srv).bytes_in_use == 0
    finally:
        V.vdi_server_destroy(srv)


def test_replaced_vdi_is_freed_after_its_generation(V, ctx):
    """A slot's VDI replaced while its generation is still queued: its memory is not
    handed to the images of the views that follow, so the late writes miss them."""
    n, w, h, ns = 64, 640, 360, 12
    vol = torch.from_numpy(S.blobs_volume(n, seed=2)).cuda()
    bmin, bmax = np.zeros(3), np.ones(3)
    co = S.orbit_camera(bmin, bmax, w / h, el_deg=15.0)
    kn, cam_o = S.tf_knots("dense"), V.camera(co.view, co.proj)
    cam = V.camera(*(lambda c: (c.view, c.proj))(S.orbit_camera(bmin, bmax, w / h, az_deg=20.0, el_deg=15.0)))
    args = (vol, bmin, bmax, kn, cam_o, w, h, ns, 0.02, 1 / n, 1 / n, V.VDI_F32)
    ref = torch.zeros((h, w, 4), device="cuda")
    vdi = V.vdi_generate(ctx, *args)
    V.vdi_render(vdi, cam, w, h, 1, 1, ref)
    torch.cuda.synchronize()
    srv = V.vdi_server_create(ctx, budget_bytes=1 << 30, n_slots=1)
    try:
        side = torch.cuda.Stream()
        with torch.cuda.stream(side):
            torch.cuda._sleep(1_000_000_000)  # half a second
        V.vdi_server_generate(srv, 0, *args, stream=side)
        V.vdi_server_set_vdi(srv, 0, vdi)  # the first version dies with its generation queued
        tickets = [V.vdi_server_submit(srv, V.view_request(0, cam, w, h, out_fmt=V.VDI_F32)) for _ in range(30)]
        assert all(V.vdi_server_wait(srv, t, 30.0).status == 0 for t in tickets)
        torch.cuda.synchronize()  # the late generation has run
        for t in tickets:
            out = torch.zeros_like(ref)
            V.vdi_server_read(srv, t, out)
            assert torch.equal(out, ref)
            V.vdi_server_release(srv, t)
    finally:
        V.vdi_server_destroy(srv)


def test_server_generates_small_vdis_from_recorded_samples(V, ctx):
    """A VDI of fewer tiles than the GPU holds warps takes little scratch, which the
    server grants: its generation takes as long as vdi_generate's (sampled at every
    gamma it would take some six times as long)."""
    n, w, h, ns = 256, 64, 64, 20
    vol = torch.from_numpy(S.value_noise_volume(n, seed=5, dtype=np.uint16)).cuda()
    bmin, bmax = np.zeros(3), np.ones(3)
    co = S.orbit_camera(bmin, bmax, 1.0, el_deg=20.0)
    args = (vol, bmin, bmax, S.tf_knots("sparse"), V.camera(co.view, co.proj), w, h, ns, 0.0, 1 / n, 1 / n, V.VDI_F32)
    srv = V.vdi_server_create(ctx, budget_bytes=1 << 30, n_slots=1)
    try:
        side = torch.cuda.Stream()

        def ms(call):
            best = 1e9
            for _ in range(5):
                a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
                a.record(side)
                call()
                b.record(side)
                torch.cuda.synchronize()
                best = min(best, a.elapsed_time(b))
            return best

        direct = ms(lambda: V.vdi_destroy(V.vdi_generate(ctx, *args, stream=side, adaptive=True)))
        served = ms(lambda: V.vdi_server_generate(srv, 0, *args, stream=side, adaptive=True))
        assert served < 2.5 * direct, (served, direct)
    finally:
        V.vdi_server_destroy(srv)
