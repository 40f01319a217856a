"""The skip field of volumes of more than 152 tiles of 32 x 24 x 24 cells, whose construction
takes two launches (the blocks' distances first) instead of one: leaping must not change an
image, as for the smaller volumes. Sizes with remainders on every axis, several 32-block words
and several 16-row tiles of blocks; the last size that takes one launch on this shape beside the
first that takes two; volumes that are almost empty, so that leaps come from far blocks."""

import numpy as np
import pytest

from phantoms import camera_array, orbit_camera
from tests.gpu_util import torch_cuda
from tests.test_gpu_skip_field import _sparse_volume, _table

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return torch_cuda()


def _tiles(dims):
    nx, ny, nz = (n - 1 for n in dims)
    return -(-nx // 32) * -(-ny // 24) * -(-nz // 24)


CASES = [
    # dims, spacing, step, blobs, more than one launch
    ((150, 169, 97), (1.0, 1.0, 1.0), 0.5, 6, False),
    ((151, 173, 97), (1.0, 1.0, 1.7), 0.5, 6, True),
    ((263, 150, 141), (1.0, 1.0, 1.0), 0.35, 9, True),
    ((263, 150, 141), (1.0, 1.0, 1.0), 1.0, 0, True),
    ((41, 700, 60), (1.0, 1.0, 1.0), 0.5, 5, True),
    ((300, 130, 121), (0.7, 1.0, 1.3), 2.5, 40, True),
]


@pytest.mark.parametrize("dims,spacing,step,blobs,two", CASES)
@pytest.mark.parametrize("brick", [8, 16])
def test_leaps_are_neutral(torch, dims, spacing, step, blobs, two, brick):
    import paper_2605_19737_gb300 as pkg
    assert (_tiles(dims) > 152) == two
    vol = _sparse_volume(dims, sum(dims), blobs)
    some = 0
    with pkg.Context(0) as ctx:
        vid = ctx.load_volume(vol, spacing)
        ctx.set_brick_size(vid, brick)
        ctx.precompute_morphology(vid)
        ctx.set_tissue_params(vid, _table(256), shading=1, grad_mod=0, step_vox=step, et_threshold=0.9)
        for W, H in ((96, 80), (470, 440)):  # several lanes per ray, and one
            cams = camera_array([orbit_camera(dims, spacing, az, el, width=W, height=H) for az, el in
                                 ((0.0, 0.0), (33.0, 21.0), (200.0, -40.0), (90.0, 80.0))])
            inside = cams[1].copy()  # a camera inside the volume
            inside[:3] = [0.4 * n * s for n, s in zip(dims, spacing)]
            cams = np.concatenate([cams, inside[None]])
            full = ctx.render(vid, cams, W, H, skip_empty=False)
            assert torch.equal(full, ctx.render(vid, cams, W, H))
            for i in range(len(cams)):  # (one view at a time has the fewest rays)
                assert torch.equal(full[i], ctx.render(vid, cams[i], W, H)[0])
            ctr, bctr = pkg.new_counters(0), pkg.new_counters(0)
            assert torch.equal(full, ctx.render(vid, cams, W, H, counters=ctr))
            views = [torch.zeros((H, W, 4), device="cuda") for _ in cams]
            bid = ctx.batch_create([(vid, cams[i], views[i], W, H) for i in range(len(cams))])
            ctx.batch_render(bid)
            ctx.synchronize()
            assert torch.equal(full, torch.stack(views))
            ctx.batch_render(bid, counters=bctr)
            ctx.synchronize()
            assert torch.equal(full, torch.stack(views)) and torch.equal(ctr, bctr)
            ctx.batch_free(bid)
            some += float(full[..., 3].max()) > 0.0
    assert blobs == 0 or some == 2
