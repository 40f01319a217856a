"""Launches that count samples, and batches, at sizes on both sides of the line below which
their kernels take more registers, and of CTAs of fewer warps: the image and the ray state are
those of the leaping kernels bit for bit, the counters the sums of the per-ray counts, and a
batch counts what single renders count."""

import numpy as np
import pytest

from phantoms import camera_array, orbit_camera
from tests.gpu_util import torch_cuda

pytestmark = pytest.mark.gpu

DIMS, SP = (61, 50, 43), (1.0, 1.0, 1.2)
# the line is 28 warps for each of 152 SMs, 136,192 rays: 369 x 369 lies below it, 370 x 369 above
SIZES = [(1, 1), (5, 3), (33, 17), (64, 75), (70, 70), (100, 100), (140, 140), (369, 369), (370, 369)]


@pytest.fixture(scope="module")
def torch():
    return torch_cuda()


def _volume(ctx, derived, brick):
    if not derived:
        ctx.set_derived_budget(0)
    vol = np.random.default_rng(3).random(DIMS[::-1], dtype=np.float32)
    vol[:, :, :20] *= 0.4  # empty under the table
    vid = ctx.load_volume(vol, SP)
    ctx.set_brick_size(vid, brick)
    ctx.precompute_morphology(vid)
    tf = np.zeros((1, 256, 4), np.float32)
    tf[0, 128:, 3] = 0.02
    tf[0, :, :3] = (0.9, 0.5, 0.2)
    ctx.set_tissue_params(vid, tf, shading=1, grad_mod=0, gamma=0.4, kappa_ref=0.05)
    return vid


@pytest.mark.parametrize("derived,brick", [(True, 4), (True, 8), (True, 16), (False, 8)])
@pytest.mark.parametrize("W,H", SIZES)
def test_few_rays(torch, derived, brick, W, H):
    import paper_2605_19737_gb300 as pkg
    cams = camera_array([orbit_camera(DIMS, SP, 40.0, 25.0, width=W, height=H)])
    with pkg.Context(0) as ctx:
        vid = _volume(ctx, derived, brick)
        st = [torch.zeros((1, H, W, 2), device="cuda") for _ in range(2)]
        want = ctx.render(vid, cams, W, H, ray_state=st[0])
        for pw, warps in ((4, 4), (16, 8), (8, 2)):
            ctr, per_ray = pkg.new_counters(0), torch.zeros((1, H, W, 2), dtype=torch.int32, device="cuda")
            img = ctx.render(vid, cams, W, H, counters=ctr, ray_samples=per_ray, packet_w=pw, warps_per_block=warps)
            state = ctx.render(vid, cams, W, H, counters=pkg.new_counters(0), ray_state=st[1])
            ctx.synchronize()
            assert torch.equal(img, want) and torch.equal(state, want)
            assert torch.equal(st[0].view(torch.int32), st[1].view(torch.int32))
            assert [int(x) for x in per_ray.long().sum((0, 1, 2))] == [int(ctr[1]), int(ctr[2])]
        if W > 1:
            assert 0 < int(ctr[2]) < int(ctr[1])
        out = torch.zeros((H, W, 4), device="cuda")
        bid = ctx.batch_create([(vid, cams[0], out, W, H)])
        for pw, warps in ((8, 8), (4, 3), (32, 1)):
            for kw in (dict(), dict(graph=True), dict(skip_empty=False), dict(counters=pkg.new_counters(0))):
                out.zero_()
                ctx.batch_render(bid, packet_w=pw, warps_per_block=warps, **kw)
                ctx.synchronize()
                assert torch.equal(out, want[0])
            assert torch.equal(kw["counters"], ctr)


@pytest.mark.parametrize("gamma,W,H", [(0.0, 400, 340), (0.0, 400, 344), (0.4, 896, 920), (0.4, 896, 928)])
def test_batch_line(torch, gamma, W, H):
    """Batches on both sides of the line between their kernels: 28 packets of 8 x 4 rays per SM
    (4256) without a curvature term, 170 (25840) with one; and one that crosses it by an update."""
    import paper_2605_19737_gb300 as pkg
    packets = -(-W // 8) * -(-H // 4)
    line = 152 * (170 if gamma else 28)
    assert abs(packets - line) < 300
    cams = camera_array([orbit_camera(DIMS, SP, 40.0, 25.0, width=W, height=H)])
    tf = np.zeros((1, 256, 4), np.float32)
    tf[0, 128:] = (0.9, 0.5, 0.2, 0.02)
    with pkg.Context(0) as ctx:
        vid = _volume(ctx, True, 8)
        out = torch.zeros((H, W, 4), device="cuda")
        bid = ctx.batch_create([(vid, cams[0], out, W, H)])  # with a curvature term
        for g in (0.4, gamma, 0.4):
            ctx.set_tissue_params(vid, tf, shading=1, grad_mod=0, gamma=g, kappa_ref=0.05)
            ctx.batch_update(bid)
            want = ctx.render(vid, cams, W, H)[0]
            for kw in (dict(), dict(graph=True), dict(graph=True, packet_w=4, warps_per_block=4)):
                out.zero_()
                ctx.batch_render(bid, **kw)
                ctx.synchronize()
                assert torch.equal(out, want)
