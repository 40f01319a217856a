"""The selection network of the 3x3x3 median at the places it can go wrong: volumes smaller
than a warp's 30 voxels, strips of four rows and chunks of sixteen planes and one past
them, many equal values, infinities, signed zeros and NaNs. The result is an element of
the neighbourhood, so it equals numpy's exactly. With NaNs the numbers sort first; with 14
or more of them the neighbour at (-1, -1, -1) is returned."""

import numpy as np
import pytest

from tests.gpu_util import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return torch_cuda()


def _median27(v):
    n = v.shape
    idx = [np.clip(np.arange(m)[:, None] + np.array([-1, 0, 1]), 0, m - 1) for m in n]
    w = v[idx[0][:, None, None, :, None, None], idx[1][None, :, None, None, :, None],
          idx[2][None, None, :, None, None, :]].reshape(*n, 27)
    s = np.sort(w, -1)  # NaNs last
    med = s[..., 13]
    return np.where(np.isnan(med), w[..., 0], med)


@pytest.mark.parametrize("dims", [(2, 2, 2), (3, 5, 2), (29, 4, 16), (30, 5, 17), (31, 16, 15), (33, 17, 33),
                                  (61, 15, 18), (64, 18, 32), (7, 33, 50)])
@pytest.mark.parametrize("kind", ["noise", "few", "special"])
def test_median(torch, dims, kind):
    import paper_2605_19737_gb300 as pkg
    rng = np.random.default_rng(sum(dims))
    nx, ny, nz = dims
    base = rng.random((nz, ny, nx), dtype=np.float32)
    v = base.copy()
    if kind == "few":
        v = rng.integers(0, 4, v.shape).astype(np.float32) / 3.0
    elif kind == "special":
        v = rng.normal(size=v.shape).astype(np.float32)
        pick = rng.random(v.shape)
        v[pick < 0.1] = np.inf
        v[(pick > 0.1) & (pick < 0.2)] = -np.inf
        v[(pick > 0.2) & (pick < 0.3)] = 0.0
        v[(pick > 0.3) & (pick < 0.4)] = -0.0
        v[(pick > 0.4) & (pick < 0.8)] = np.nan
    with pkg.Context(0) as ctx:
        vid = ctx.load_volume(base, (1.0, 1.0, 1.0))
        ctx.set_normalized(vid, torch.from_numpy(v).cuda())
        ctx.prefilter(vid, "median")
        got = ctx.get_normalized(vid)
        ctx.synchronize()
    np.testing.assert_array_equal(got.cpu().numpy(), _median27(v))
