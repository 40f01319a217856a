"""Vesselness on a volume whose plane walks are twelve planes with a last one of seven, and whose
CTAs at the far x and y ends are partly filled: the queue of voxels to decompose is drained after
a clipped walk."""

import numpy as np
import pytest

import oracle
from phantoms import volumes
from tests.gpu_util import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sigmas", [(1.0,), (1.5, 2.5)])
def test_vesselness_short_last_walk(sigmas):
    torch = torch_cuda()
    import paper_2605_19737_gb300 as pkg
    vol = volumes.vessel_phantom((330, 251, 43), seed=51)
    with pkg.Context(0) as ctx:
        vid = ctx.load_volume(torch.from_numpy(vol).cuda())
        ctx.precompute_morphology(vid, sigmas)
        got = ctx.get_vesselness(vid).cpu().numpy().astype(np.float64)
    V, _, amb = oracle.frangi(oracle.normalize(vol), sigmas)
    assert V.max() > 0.3
    assert (np.abs(got - V)[amb == 0] <= 1e-4).all()
