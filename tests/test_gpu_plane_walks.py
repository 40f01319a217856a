"""Kernels whose CTAs walk several planes along z, on volumes wide enough that the walks
are longer than one plane and the last one is shorter (small volumes get one plane per
CTA, which the other tests cover), and the Gaussian at radii outside the unrolled ones."""

import numpy as np
import pytest

import oracle
from phantoms import camera_array, orbit_camera, volumes
from tests.gpu_util import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return torch_cuda()


@pytest.fixture()
def ctx(torch):
    import paper_2605_19737_gb300 as pkg
    with pkg.Context(0) as c:
        yield c


@pytest.mark.parametrize("sigma", [0.2, 0.3, 1.1, 1.5, 2.3, 7.9])  # radii 1, 2, 5, 6, 10, 32
def test_gauss_any_radius(ctx, torch, sigma):
    vol = volumes.head_phantom((37, 29, 23), seed=7)
    vid = ctx.load_volume(torch.from_numpy(vol).cuda())
    before = ctx.get_normalized(vid).cpu().numpy().astype(np.float64)
    ctx.prefilter(vid, "gauss", sigma)
    got = ctx.get_normalized(vid).cpu().numpy()
    # three passes of 2R + 1 fmaf on values in [0, 1] with weights rounded once and summing to 1
    tol = 3 * (2 * np.ceil(4 * sigma) + 2) * 2.0 ** -24
    np.testing.assert_allclose(got, oracle.gauss_smooth(before, sigma), rtol=0, atol=tol)


def test_median_long_walk(ctx, torch):
    """512x512x21: walks of nine planes; checked on both ends of every axis."""
    v = np.random.default_rng(2).random((21, 512, 512), dtype=np.float32)
    vid = ctx.load_volume(torch.from_numpy(v).cuda())
    v = ctx.get_normalized(vid).cpu().numpy()
    ctx.prefilter(vid, "median")
    got = ctx.get_normalized(vid).cpu().numpy()
    for ys in (slice(0, 20), slice(-20, None)):
        for xs in (slice(0, 40), slice(-40, None)):
            want = oracle.median3(v[:, ys, xs].astype(np.float64)).astype(np.float32)
            iy = slice(0, 19) if ys.start == 0 else slice(1, None)  # without the crop's own border
            ix = slice(0, 39) if xs.start == 0 else slice(1, None)
            np.testing.assert_array_equal(got[:, ys, xs][:, iy, ix], want[:, iy, ix])


def test_vesselness_long_walk(ctx, torch):
    """320x256x40: walks of ten planes."""
    vol = volumes.vessel_phantom((320, 256, 40), seed=51)
    vid = ctx.load_volume(torch.from_numpy(vol).cuda())
    ctx.precompute_morphology(vid, (1.0,))
    got = ctx.get_vesselness(vid).cpu().numpy().astype(np.float64)
    V, _, amb = oracle.frangi(oracle.normalize(vol), (1.0,))
    assert V.max() > 0.3
    assert (np.abs(got - V)[amb == 0] <= 1e-4).all()


def test_voxel_gradient_long_walk(torch):
    """256x256x33: walks of twelve planes and a shorter one. The derived path's gather against the per-sample
    stencils' direct scatter: the same linear map, so with a table without knots the two
    differ by float32 rounding of samples and sums (of the order of 1e-5); a plane taken
    wrongly changes 1/33 of the voxels."""
    import paper_2605_19737_gb300 as pkg
    dims, W, H = (256, 256, 33), 160, 120
    vol = volumes.head_phantom(dims, seed=5)
    x = np.arange(64, dtype=np.float32) / 63.0
    tf = np.stack([x, 1.0 - x, 0.5 * x, 0.01 + 0.02 * x], -1)[None].astype(np.float32)
    cams = camera_array([orbit_camera(dims, (1.0, 1.0, 1.3), 20.0, 60.0, width=W, height=H)])
    g = torch.rand((1, H, W, 4), generator=torch.Generator(device="cuda").manual_seed(9), device="cuda")
    out = []
    for derived in (True, False):
        with pkg.Context(0) as c:
            if not derived:
                c.set_derived_budget(0)
            vid = c.load_volume(vol, (1.0, 1.0, 1.3))
            c.precompute_morphology(vid)
            c.set_tissue_params(vid, tf, tf_mode=0, grad_mod=0, shading=0, gamma=0.0, kappa_ref=0.05, w_max=3.0)
            out.append(c.render_backward(vid, cams, W, H, g)[2].double())
            c.synchronize()
    assert float(out[1].abs().max()) > 0
    assert float((out[0] - out[1]).norm() / out[1].norm()) <= 1e-4
