"""Renders of volumes whose skip field was given up for another buffer (or that never had one):
the same images, ray states and counts, in single renders and in batches made before."""

import numpy as np
import pytest

from phantoms import camera_array, orbit_camera
from tests.gpu_util import torch_cuda

pytestmark = pytest.mark.gpu

DIMS, SP = (61, 50, 43), (1.0, 1.0, 1.2)


@pytest.fixture(scope="module")
def torch():
    return torch_cuda()


def _images(torch, pkg, ctx, vid, cams, sizes, batches):
    out = []
    for (W, H), cam in zip(sizes, cams):
        st, ctr = torch.zeros((1, H, W, 2), device="cuda"), pkg.new_counters(0)
        out += [ctx.render(vid, cam, W, H, ray_state=st), st.view(torch.int32),  # (sample index as integer bits)
                ctx.render(vid, cam, W, H, counters=ctr),
                ctx.render(vid, cam, W, H)]
        ctx.synchronize()
        out.append(ctr[:3].clone())  # rays, samples, evaluated samples; what is interpolated differs
    for bid, views in batches:
        for kw in (dict(), dict(graph=True), dict(packet_w=4, warps_per_block=2)):
            for v in views:
                v.zero_()
            ctx.batch_render(bid, **kw)
            ctx.synchronize()
            out += [v.clone() for v in views]
    return [o.cpu() for o in out]


@pytest.mark.parametrize("derived", [True, False])
def test_field_given_up_for_another_buffer(torch, derived):
    import paper_2605_19737_gb300 as pkg
    sizes = [(45, 37), (370, 369), (470, 460)]
    cams = [camera_array([orbit_camera(DIMS, SP, 40.0, 25.0, width=W, height=H)]) for W, H in sizes]
    vol = np.random.default_rng(3).random(DIMS[::-1], dtype=np.float32)
    vol[:, :, :20] *= 0.4  # empty under the table
    tf = np.zeros((1, 256, 4), np.float32)
    tf[0, 128:, 3] = 0.02
    tf[0, :, :3] = (0.9, 0.5, 0.2)
    with pkg.Context(0) as ctx:
        if not derived:
            ctx.set_derived_budget(0)
        vids = []
        for k in range(2):
            vids.append(ctx.load_volume(vol if k == 0 else vol[::-1].copy(), SP))
            ctx.precompute_morphology(vids[k])
            ctx.set_tissue_params(vids[k], tf, shading=1, grad_mod=0, gamma=0.4, kappa_ref=0.05)
        views = [torch.zeros((H, W, 4), device="cuda") for W, H in sizes]
        batches = [(ctx.batch_create([(vids[(k + i) % 2], cams[i][0], views[i], *sizes[i]) for i in range(3)]), views)
                   for k in range(2)]
        args = (torch, pkg, ctx, vids[0], cams, sizes, batches)
        want = _images(*args)
        used = ctx.memory_used()
        cells = 2 * np.prod([n - 1 for n in DIMS])
        ctx.set_memory_limit(used + 1024)  # no room for the gradient's buffers but the fields'
        H, W = sizes[0][1], sizes[0][0]
        g = torch.ones((1, H, W, 4), device="cuda")
        with pytest.raises(pkg.VRError):
            ctx.render_backward(vids[0], cams[0], W, H, g)  # 10 floats per voxel and the table's copies
        ctx.tissue_histogram(vids[0])
        assert ctx.memory_used() == used  # nothing was given up for a call that fails all the same
        ctx.reduce_minmax(torch.zeros(1 << 22, device="cuda"))  # no more scratch than it had
        big = ctx.load_volume(np.random.default_rng(1).random((16, 16, 16), dtype=np.float32))
        assert ctx.memory_used() < used - 4 * cells
        for a, b in zip(_images(*args), want):
            assert torch.equal(a, b)
        ctx.free_volume(big)
        ctx.set_memory_limit(0)
        ctx.render_backward(vids[0], cams[0], W, H, g)
        for vid in vids:
            ctx.precompute_morphology(vid)
        for a, b in zip(_images(*args), want):
            assert torch.equal(a, b)


def test_no_precompute(torch):
    """A volume that only got its largest gradient has neither derived bricks nor a field."""
    import paper_2605_19737_gb300 as pkg
    W, H = 100, 80
    cams = camera_array([orbit_camera(DIMS, SP, 40.0, 25.0, width=W, height=H)])
    vol = np.random.default_rng(3).random(DIMS[::-1], dtype=np.float32)
    vol[:, :, :20] *= 0.4
    tf = np.zeros((1, 256, 4), np.float32)
    tf[0, 128:] = (0.9, 0.5, 0.2, 0.02)
    imgs = []
    for precompute in (True, False):
        with pkg.Context(0) as ctx:
            ctx.set_derived_budget(0)
            vid = ctx.load_volume(vol, SP)
            if precompute:
                ctx.precompute_morphology(vid)
                gmax = ctx.get_norm(vid)[2]
            else:
                ctx.set_gmax(vid, gmax)
            ctx.set_tissue_params(vid, tf, shading=1, gamma=0.4, kappa_ref=0.05)
            out = torch.zeros((H, W, 4), device="cuda")
            bid = ctx.batch_create([(vid, cams[0], out, W, H)])
            ctx.batch_render(bid)
            imgs += [ctx.render(vid, cams, W, H)[0].cpu(), out.cpu()]
    assert float(imgs[0][..., 3].max()) > 0.1
    assert all(torch.equal(i, imgs[0]) for i in imgs)
