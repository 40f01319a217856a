"""Freed buffers kept for reuse: not counted as used, safe to reuse by another context or
thread and after a context changed its stream, never shared by two volumes, and given
back with the last context."""

import numpy as np
import pytest

from phantoms import camera_array, orbit_camera, volumes, workloads
from tests.gpu_util import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    return torch_cuda()


def _open(ctx, vol, case, dims):
    vid = ctx.load_volume(vol, (1.0, 1.0, 1.0))
    ctx.precompute_morphology(vid)
    ctx.set_tissue_params(vid, case["tf"][:1], **dict(case["params"], tf_mode=0))
    return vid


@pytest.mark.parametrize("switch", [False, True])
def test_reopened_studies(torch, switch):
    import paper_2605_19737_gb300 as pkg
    case = workloads.scaled_brainweb((40, 48, 36))
    sizes = [(40, 48, 36), (40, 48, 36), (33, 20, 51), (40, 48, 36), (41, 48, 36)]
    want, used = [], []
    for k, dims in enumerate(sizes):  # each in a context of its own
        with pkg.Context(0) as ctx:
            vid = _open(ctx, volumes.brainweb_phantom(dims, seed=k), case, dims)
            cams = camera_array([orbit_camera(dims, (1, 1, 1), 20.0 * k, 10.0, width=64, height=48)])
            want.append(ctx.render(vid, cams, 64, 48).cpu())
            used.append(ctx.memory_used())
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    with pkg.Context(0) as ctx:
        base = ctx.memory_used()
        for k, dims in enumerate(sizes):
            if switch:
                ctx.set_stream(streams[k & 1])
            vid = _open(ctx, volumes.brainweb_phantom(dims, seed=k), case, dims)
            cams = camera_array([orbit_camera(dims, (1, 1, 1), 20.0 * k, 10.0, width=64, height=48)])
            img = ctx.render(vid, cams, 64, 48)
            ctx.synchronize()
            assert torch.equal(img.cpu(), want[k])
            assert ctx.memory_used() <= max(used)
            ctx.free_volume(vid)
        # two volumes of one size open at once, after both buffers became spare
        dims = sizes[0]
        a = _open(ctx, volumes.brainweb_phantom(dims, seed=0), case, dims)
        b = _open(ctx, volumes.brainweb_phantom(dims, seed=1), case, dims)
        cams = [camera_array([orbit_camera(dims, (1, 1, 1), 20.0 * k, 10.0, width=64, height=48)]) for k in (0, 1)]
        ia, ib = ctx.render(a, cams[0], 64, 48), ctx.render(b, cams[1], 64, 48)
        ctx.synchronize()
        assert torch.equal(ia.cpu(), want[0]) and torch.equal(ib.cpu(), want[1])
        ctx.free_volume(a)
        ctx.free_volume(b)
        # a limit is all there for what is asked for
        ctx.set_memory_limit(base + max(used))
        for k, dims in enumerate(sizes):
            vid = _open(ctx, volumes.brainweb_phantom(dims, seed=k), case, dims)
            cams = camera_array([orbit_camera(dims, (1, 1, 1), 20.0 * k, 10.0, width=64, height=48)])
            img = ctx.render(vid, cams, 64, 48)
            ctx.synchronize()
            assert torch.equal(img.cpu(), want[k])
            ctx.free_volume(vid)


def test_contexts_share_freed_buffers(torch):
    """Contexts on several threads and streams open and close studies of the same sizes at
    once: every image is the one a context alone gives; with the last context everything
    is given back."""
    import gc
    import threading

    import paper_2605_19737_gb300 as pkg
    case = workloads.scaled_brainweb((40, 48, 36))
    dims = (40, 48, 36)
    vols = [volumes.brainweb_phantom(dims, seed=k) for k in range(4)]
    cams = camera_array([orbit_camera(dims, (1, 1, 1), 30.0, 10.0, width=96, height=80)])
    want = []
    for v in vols:
        with pkg.Context(0) as ctx:
            want.append(ctx.render(_open(ctx, v, case, dims), cams, 96, 80).cpu())
    bad = []

    def work(t):
        try:
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                for rep in range(6):
                    with pkg.Context(0, stream=stream) as ctx:
                        for k in range(4):
                            j = (k + t + rep) % 4
                            vid = _open(ctx, vols[j], case, dims)
                            img = ctx.render(vid, cams, 96, 80)
                            ctx.synchronize()
                            if not torch.equal(img.cpu(), want[j]):
                                bad.append((t, rep, j))
                            ctx.free_volume(vid)
        except Exception as e:  # reported by the main thread
            bad.append(repr(e))

    ts = [threading.Thread(target=work, args=(t,)) for t in range(4)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not bad, bad[:3]
    gc.collect()
    torch.cuda.empty_cache()
    free0 = torch.cuda.mem_get_info()[0]
    big = np.zeros((128, 256, 256), np.float32)
    big[64] = 1.0
    with pkg.Context(0) as ctx:
        vid = ctx.load_volume(big, (1.0, 1.0, 1.0))
        ctx.precompute_morphology(vid)
        ctx.synchronize()
        ctx.free_volume(vid)
    assert torch.cuda.mem_get_info()[0] >= free0 - (64 << 20)
