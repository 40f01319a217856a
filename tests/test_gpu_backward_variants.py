"""The backward's specialised kernels against the general one.

A launch that wants fewer gradients, or whose table is 1D, runs a kernel with the rest
compiled out; what it does compute must equal the general kernel's (which the oracle
tests cover). Both add the same float32 terms, only in another order: an entry's sum is a
few hundred additions per private copy plus the copies' sum, so the two differ by at most
~264 * 2^-24 = 1.6e-5 of the sum of magnitudes; 2e-5 of the norm is asserted on gradients
whose terms do not cancel (a positive upstream gradient)."""

import numpy as np
import pytest

from phantoms import camera_array, orbit_camera, volumes
from tests.gpu_util import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return torch_cuda()


def _rel(a, b):
    a, b = a.double(), b.double()
    return float((a - b).norm() / b.norm())


def _scene(ctx, torch, mode, gamma, derived, brick, W, H, n, corr=0.0):
    dims, sp = (49, 40, 37), (1.0, 1.0, 1.3)
    if not derived:
        ctx.set_derived_budget(0)
    vid = ctx.load_volume(volumes.head_phantom(dims, seed=5), sp)
    ctx.set_brick_size(vid, brick)
    ctx.precompute_morphology(vid, (1.0,))
    rng = np.random.default_rng(3)
    rows = 1 if mode == 0 else 16
    tf = rng.random((rows, 64, 4)).astype(np.float32) * np.array([1, 1, 1, 0.15], np.float32)
    tf[:, :20, 3] = 0.0  # empty space too
    ctx.set_tissue_params(vid, tf, tf_mode=mode, grad_mod=1 if mode == 0 else 0, shading=1, gamma=gamma,
                          kappa_ref=0.05, w_max=3.0, opacity_ref_step=corr)
    cams = camera_array([orbit_camera(dims, sp, 30.0 + 100.0 * i, 20.0 - 30.0 * i, width=W, height=H)
                         for i in range(n)])
    g = torch.rand((n, H, W, 4), generator=torch.Generator(device="cuda").manual_seed(9), device="cuda")
    return vid, cams, g


@pytest.mark.parametrize("mode", [0, 1, 2])
@pytest.mark.parametrize("gamma", [0.0, 0.6])
@pytest.mark.parametrize("derived,brick", [(True, 4), (True, 8), (True, 16), (False, 8)])
@pytest.mark.parametrize("stated", [False, True])
def test_fewer_gradients_same_values(torch, mode, gamma, derived, brick, stated):
    import paper_2605_19737_gb300 as pkg
    W, H, n = 52, 39, 2
    with pkg.Context(0) as ctx:
        vid, cams, g = _scene(ctx, torch, mode, gamma, derived, brick, W, H, n)
        st = torch.empty((n, H, W, 2), device="cuda") if stated else None
        if stated:
            ctx.render(vid, cams, W, H, ray_state=st)
        full = ctx.render_backward(vid, cams, W, H, g, ray_state=st)
        tf_only = ctx.render_backward(vid, cams, W, H, g, ray_state=st, want_params=False, want_volume=False)
        no_par = ctx.render_backward(vid, cams, W, H, g, ray_state=st, want_params=False)
        no_vol = ctx.render_backward(vid, cams, W, H, g, ray_state=st, want_volume=False)
        ctx.synchronize()
        assert float(full[0].abs().max()) > 0 and float(full[2].abs().max()) > 0
        for other in (tf_only, no_par, no_vol):
            assert _rel(other[0], full[0]) <= 2e-5
        assert _rel(no_vol[1], full[1]) <= 2e-5
        assert _rel(no_par[2], full[2]) <= 2e-5


# both sides of every line between 16, 8, 4, 2 and 1 lanes per ray
@pytest.mark.parametrize("W,H", [(9, 5), (75, 80), (95, 64), (160, 175), (180, 160), (300, 300), (303, 300),
                                 (384, 320), (390, 320)])
@pytest.mark.parametrize("mode,gamma,corr", [(0, 0.0, 0.0), (1, 0.6, 0.0), (2, 0.6, 0.8)])
def test_lanes_per_ray(torch, W, H, mode, gamma, corr):
    """With a recorded ray state a small launch gives each ray several lanes; without one
    it re-marches with one lane per ray. Same terms, another order."""
    import paper_2605_19737_gb300 as pkg
    with pkg.Context(0) as ctx:
        vid, cams, g = _scene(ctx, torch, mode, gamma, True, 8, W, H, 1, corr)
        st = torch.empty((1, H, W, 2), device="cuda")
        ctx.render(vid, cams, W, H, ray_state=st)
        lanes = ctx.render_backward(vid, cams, W, H, g, ray_state=st)
        tf_only = ctx.render_backward(vid, cams, W, H, g, ray_state=st, want_params=False, want_volume=False)
        one = ctx.render_backward(vid, cams, W, H, g)
        ctx.synchronize()
        assert float(one[2].abs().max()) > 0
        for a, b in zip(lanes, one):
            assert _rel(a, b) <= 2e-5
        assert _rel(tf_only[0], one[0]) <= 2e-5
