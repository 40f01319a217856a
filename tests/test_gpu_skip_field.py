"""The skip field: leaping over empty space must not change an image.

A sample in a cell the field marks empty has opacity exactly 0, so a render that leaps
equals the one that visits every sample (skip_empty=False) bit for bit, and the
counting variant (which walks brick by brick) equals the leaping one. Sizes cross the
edges of the field's construction: 32-cell words, 4-cell blocks, the 24- and 16-row
tiles of the distance kernels, rows shorter than a word; steps from a hundredth of a
voxel to several voxels; tables of 2 to 4096 columns."""

import numpy as np
import pytest

from phantoms import camera_array, orbit_camera
from tests.gpu_util import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return torch_cuda()


def _sparse_volume(dims, seed, blobs):
    """Zero background with a few bright blobs and single bright voxels."""
    rng = np.random.default_rng(seed)
    nx, ny, nz = dims
    v = 0.02 * rng.random((nz, ny, nx))
    for _ in range(blobs):
        c = [rng.integers(0, n) for n in (nz, ny, nx)]
        r = int(rng.integers(0, 3))
        v[tuple(slice(max(q - r, 0), q + r + 1) for q in c)] = 0.6 + 0.4 * rng.random()
    v.flat[0], v.flat[-1] = 0.0, 1.0
    return v.astype(np.float32)


def _table(width):
    tf = np.zeros((1, width, 4), np.float32)
    lo = width // 2 if width > 2 else 1
    tf[0, lo:, 3] = 0.2
    tf[0, :, :3] = (0.9, 0.5, 0.2)
    return tf


CASES = [
    # dims, spacing, step, table width, blobs
    ((2, 2, 2), (1.0, 1.0, 1.0), 0.05, 256, 0),
    ((5, 3, 2), (1.0, 1.0, 1.0), 0.5, 2, 1),
    ((33, 25, 17), (1.0, 1.0, 1.0), 0.5, 256, 3),
    ((34, 26, 26), (1.0, 1.3, 0.7), 0.35, 256, 4),
    ((65, 18, 50), (1.0, 1.0, 3.0), 1.0, 4096, 6),
    ((130, 49, 41), (1.0, 1.0, 1.0), 0.5, 255, 8),
    ((70, 97, 130), (0.5, 1.0, 1.0), 3.0, 64, 10),
    ((150, 60, 60), (1.0, 1.0, 1.0), 0.11, 256, 5),
]


@pytest.mark.parametrize("dims,spacing,step,width,blobs", CASES)
@pytest.mark.parametrize("derived", [True, False])
def test_leaps_are_neutral(torch, dims, spacing, step, width, blobs, derived):
    import paper_2605_19737_gb300 as pkg
    W, H = 45, 37
    cams = camera_array([orbit_camera(dims, spacing, az, el, width=W, height=H) for az, el in
                         ((0.0, 0.0), (33.0, 21.0), (200.0, -40.0))])
    inside = cams[1].copy()  # a camera inside the volume
    inside[:3] = [0.4 * n * s for n, s in zip(dims, spacing)]
    cams = np.concatenate([cams, inside[None]])
    vol = _sparse_volume(dims, sum(dims), blobs)
    with pkg.Context(0) as ctx:
        if not derived:
            ctx.set_derived_budget(0)
        vid = ctx.load_volume(vol, spacing)
        for brick in (8, 4, 16):
            ctx.set_brick_size(vid, brick)
            ctx.precompute_morphology(vid)
            ctx.set_tissue_params(vid, _table(width), shading=1, grad_mod=0, step_vox=step, et_threshold=0.9)
            full = ctx.render(vid, cams, W, H, skip_empty=False)
            leap = ctx.render(vid, cams, W, H)
            ctr = pkg.new_counters(0)
            counted = ctx.render(vid, cams, W, H, counters=ctr)
            views = [torch.empty((H, W, 4), device="cuda") for _ in cams]
            bid = ctx.batch_create([(vid, cams[i], views[i], W, H) for i in range(len(cams))])
            ctx.batch_render(bid)
            bctr = pkg.new_counters(0)
            ctx.synchronize()
            assert blobs == 0 or float(full[..., 3].max()) > 0.0
            assert torch.equal(full, leap)
            assert torch.equal(full, counted)
            assert torch.equal(full, torch.stack(views))
            ctx.batch_render(bid, counters=bctr)
            ctx.synchronize()
            assert torch.equal(ctr, bctr)
            assert torch.equal(full, torch.stack(views))
            # a batch keeps the step it was created with: the field must suit any step
            ctx.set_tissue_params(vid, _table(width), shading=1, grad_mod=0, step_vox=max(0.01, 0.2 * step),
                                  et_threshold=0.9)
            ctx.batch_render(bid)
            ctx.synchronize()
            assert torch.equal(full, torch.stack(views))
            ctx.batch_free(bid)
        # a table that empties everything, then one that opens everything again
        none = _table(width)
        none[..., 3] = 0.0
        ctx.set_tissue_params(vid, none, grad_mod=0, step_vox=step)
        assert float(ctx.render(vid, cams, W, H).abs().max()) == 0.0
        every = _table(width)
        every[..., 3] = 0.01
        ctx.set_tissue_params(vid, every, grad_mod=0, step_vox=step)
        assert torch.equal(ctx.render(vid, cams, W, H), ctx.render(vid, cams, W, H, skip_empty=False))


# images on both sides of every line between 16, 8, 4, 2 and 1 lanes per ray
SIZES = [(16, 8), (61, 67), (100, 61), (150, 160), (190, 149), (300, 301), (330, 307), (420, 430), (470, 460)]


@pytest.mark.parametrize("W,H", SIZES)
@pytest.mark.parametrize("derived", [True, False])
def test_lanes_per_ray_are_neutral(torch, W, H, derived):
    """The image and the ray state of a small launch (several lanes per ray) equal those
    of the one-lane kernel, which a render with counters always takes, bit for bit."""
    import paper_2605_19737_gb300 as pkg
    dims, sp = (61, 50, 43), (1.0, 1.0, 1.2)
    cams = camera_array([orbit_camera(dims, sp, 40.0, 25.0, width=W, height=H)])
    rng = np.random.default_rng(W)
    vol = rng.random(dims[::-1], dtype=np.float32)
    tf = _table(256)
    with pkg.Context(0) as ctx:
        if not derived:
            ctx.set_derived_budget(0)
        vid = ctx.load_volume(vol, sp)
        ctx.precompute_morphology(vid, (1.0,))
        for mode, et in ((0, 0.99), (0, 2.0), (2, 0.8)):
            table = np.repeat(tf, 4, 0) if mode else tf
            ctx.set_tissue_params(vid, table, tf_mode=mode, shading=1, grad_mod=0, gamma=0.4, kappa_ref=0.05,
                                  et_threshold=et, opacity_scale=30.0 if et > 1 else 1.0)
            st = [torch.zeros((1, H, W, 2), device="cuda") for _ in range(2)]
            img = ctx.render(vid, cams, W, H, ray_state=st[0])
            one = ctx.render(vid, cams, W, H, ray_state=st[1], counters=pkg.new_counters(0))
            plain = ctx.render(vid, cams, W, H, skip_empty=False)
            ctx.synchronize()
            assert float(one[..., 3].max()) > 0.5
            assert torch.equal(img, one) and torch.equal(plain, one)
            assert torch.equal(st[0].view(torch.int32), st[1].view(torch.int32))
