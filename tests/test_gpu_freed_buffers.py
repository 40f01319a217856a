"""Freed buffers on the device: a caller's graph that holds a batch launch may still be
running, on a stream the library does not know, when a volume of the batch is freed; and
another thread may be capturing meanwhile."""

import threading

import pytest

from phantoms import camera_array, orbit_camera, volumes, workloads
from tests.gpu_util import torch_cuda

pytestmark = pytest.mark.gpu

DIMS = (61, 73, 59)


@pytest.fixture(scope="module")
def torch():
    return torch_cuda()


def _open(ctx, seed, dims=DIMS):
    case = workloads.scaled_brainweb(dims)
    vid = ctx.load_volume(volumes.brainweb_phantom(dims, seed=seed), (1.0, 1.0, 1.0))
    ctx.precompute_morphology(vid)
    ctx.set_tissue_params(vid, case["tf"][:1], **dict(case["params"], tf_mode=0))
    return vid


def test_replay_on_another_stream_outlives_its_volume(torch):
    """The replay's images are those of the volume it was captured with, although the volume
    is freed while it runs and another of the same size is opened at once."""
    import paper_2605_19737_gb300 as pkg
    W, H, n = 640, 480, 24
    cams = camera_array([orbit_camera(DIMS, (1, 1, 1), 15.0 * k, 10.0, width=W, height=H) for k in range(n)])
    side, elsewhere = torch.cuda.Stream(), torch.cuda.Stream()
    with pkg.Context(0) as ctx, pkg.Context(0, stream=side) as other:
        ctx.free_volume(_open(ctx, 0))  # the library keeps freed memory from here on
        vid = _open(ctx, 0)
        outs = [torch.zeros((H, W, 4), device="cuda") for _ in range(n)]
        bid = ctx.batch_create([(vid, cams[k], outs[k], W, H) for k in range(n)])
        ctx.batch_render(bid)
        ctx.synchronize()
        want = [o.cpu() for o in outs]
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            ctx.set_stream(torch.cuda.current_stream())
            ctx.batch_render(bid)
        ctx.set_stream(torch.cuda.default_stream())
        for k in range(n):
            outs[k].zero_()
        torch.cuda.synchronize()
        with torch.cuda.stream(elsewhere):
            for _ in range(4):
                graph.replay()
        ctx.free_volume(vid)
        for c in (ctx, other):
            _open(c, 1)
        torch.cuda.synchronize()
        for o, w in zip(outs, want):
            assert torch.equal(o.cpu(), w)


def test_capture_on_another_thread_stays_valid(torch):
    """Volumes are opened and freed while another thread captures in thread-local mode."""
    import paper_2605_19737_gb300 as pkg
    x = torch.zeros(1000, device="cuda")
    torch.cuda.synchronize()
    inside, done, err = threading.Event(), threading.Event(), []
    graph = torch.cuda.CUDAGraph()

    def capture():
        try:
            with torch.cuda.graph(graph, stream=torch.cuda.Stream(), capture_error_mode="thread_local"):
                x.add_(1.0)
                inside.set()
                done.wait(60)
                x.add_(1.0)
        except Exception as e:
            err.append(e)
            inside.set()

    stream = torch.cuda.Stream()
    with pkg.Context(0, stream=stream) as ctx:
        ctx.free_volume(_open(ctx, 0))  # the library keeps freed memory from here on
        vid = _open(ctx, 0)
        t = threading.Thread(target=capture)
        t.start()
        try:
            assert inside.wait(60)
            ctx.free_volume(vid)
            ctx.free_volume(_open(ctx, 1))
        finally:
            done.set()
            t.join()
    assert not err, err
    graph.replay()
    torch.cuda.synchronize()
    assert float(x[0]) == 2.0


def test_freed_memory_is_there_for_torch(torch):
    """After a volume is freed torch can have all the memory that is free and part of what the
    library kept, while the context lives; the context then works as before."""
    import paper_2605_19737_gb300 as pkg
    dims = (200, 200, 200)
    cams = camera_array([orbit_camera(dims, (1, 1, 1), 20.0, 10.0, width=64, height=48)])
    with pkg.Context(0) as ctx:
        ctx.free_volume(_open(ctx, 0))  # the library keeps freed memory from here on
        vid = _open(ctx, 0, dims)
        want = ctx.render(vid, cams, 64, 48).cpu()
        used = ctx.memory_used()
        ctx.free_volume(vid)
        taken = used - ctx.memory_used()
        assert taken > 500 << 20
        torch.cuda.empty_cache()
        big = torch.empty(torch.cuda.mem_get_info()[0] + taken // 2, dtype=torch.uint8, device="cuda")
        del big
        torch.cuda.empty_cache()
        assert torch.equal(ctx.render(_open(ctx, 0, dims), cams, 64, 48).cpu(), want)
