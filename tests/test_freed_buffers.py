"""What the library does with freed device buffers, on a CUDA runtime without a GPU
(tests/native/fake_cuda.cpp linked with the library's host code).

A batch launch may be captured into a caller's graph and replayed on any stream, which the
library cannot see. Freed memory must not be handed out again before the whole device has
been waited for, as cudaFree does, whichever call frees it; when that wait fails, it must not
be handed out at all."""

import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2605_19737_gb300 import build as native
from paper_2605_19737_gb300 import vr as vrlib

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    native.build(debug=False)
    out = str(tmp_path_factory.mktemp("fake") / "libvr_fake.so")
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(native._nvcc())))
    # -Bsymbolic: the fake runtime, whatever CUDA runtime the process has loaded
    subprocess.run(["g++", "-std=c++17", "-O1", "-g", "-shared", "-fPIC", "-Wl,-Bsymbolic",
                    "-I" + os.path.join(cuda, "include"), "-I" + native.INCLUDE,
                    os.path.join(HERE, "native", "fake_cuda.cpp"), os.path.join(native.BUILD, "vr_api.o"), "-ldl",
                    "-o", out], check=True)
    lib = ctypes.CDLL(out)
    lib.fake_held_bytes.restype = ctypes.c_longlong
    lib.vr_last_error.restype = ctypes.c_char_p
    return lib


class Lib:
    """One context of the fake library. fail_waits: every wait fails during the calls made
    through `freeing` (as on a stream under capture, or one that the caller has destroyed)."""

    def __init__(self, lib, fail_waits=False, reopens=True):
        """reopens: a volume has been freed, after which buffers come from the pool."""
        self.lib, self.h, self.fail_waits = lib, ctypes.c_void_p(), fail_waits
        assert lib.vr_create(ctypes.byref(self.h), 0, None) == 0
        if reopens:
            self.ok(lib.vr_free_volume(self.h, self.load(3)))

    def ok(self, status):
        assert status == 0, self.lib.vr_last_error(self.h)

    def freeing(self, fn, *args):
        """fn while unknown work that uses every buffer is on the device."""
        self.lib.fake_replay()
        self.lib.fake_fail_waits(int(self.fail_waits))
        try:
            self.ok(fn(self.h, *args))
        finally:
            self.lib.fake_fail_waits(0)

    def load(self, n=12):
        vol = np.zeros((n, n, n), np.float32)
        vid = ctypes.c_int()
        self.ok(self.lib.vr_load_volume(self.h, ctypes.c_void_p(vol.ctypes.data), 1, 0, n, n, n, ctypes.c_float(1),
                                        ctypes.c_float(1), ctypes.c_float(1), ctypes.byref(vid)))
        return vid.value

    def open(self, n=12):
        vid = self.load(n)
        self.ok(self.lib.vr_precompute_morphology(self.h, vid, None, 0))
        self.params(vid)
        return vid

    def params(self, vid, width=256, call=None):
        tf = np.zeros((1, width, 4), np.float32)
        tp = vrlib.vr_tissue_params(0, width, 1, tf.ctypes.data, 0, 0, 0, 0.0, 1.0, 4.0, 0.3, 0.7, 0.2, 1.0, 0.99, 0.5,
                                    0.0)
        (call or (lambda fn, *a: self.ok(fn(self.h, *a))))(self.lib.vr_set_tissue_params, vid, ctypes.byref(tp))

    def batch(self, vid, views=3):
        img = np.zeros((8, 8, 4), np.float32)
        arr = (vrlib.vr_view * views)()
        for k in range(views):
            arr[k] = vrlib.vr_view(vid, vrlib.vr_camera(), img.ctypes.data, 8, 8)
        bid = ctypes.c_int()
        self.ok(self.lib.vr_batch_create(self.h, arr, views, ctypes.byref(bid)))
        return bid.value

    def used(self):
        n = ctypes.c_ulonglong()
        self.ok(self.lib.vr_memory_used(self.h, ctypes.byref(n)))
        return n.value

    def close(self):
        if self.h:
            self.lib.vr_destroy(self.h)
            self.h = ctypes.c_void_p()


# Each frees buffers during unknown work and then asks for buffers of the same sizes.


def _free_volume(c):
    c.open()
    c.freeing(c.lib.vr_free_volume, c.open())
    c.load()


def _free_batch(c):
    vid = c.open()
    c.freeing(c.lib.vr_batch_free, c.batch(vid))
    c.batch(vid)


def _destroy(c):
    c.open()
    with_volume = Lib(c.lib)
    with_volume.open()
    c.lib.fake_replay()
    c.lib.fake_fail_waits(int(c.fail_waits))
    with_volume.close()
    c.lib.fake_fail_waits(0)
    c.open()


def _brick_size(c):
    c.freeing(c.lib.vr_set_brick_size, c.open(30), 4)
    c.open(30)


def _wider_table(c):
    narrow, wide = c.load(), c.open()
    c.params(wide, 512, c.freeing)  # the buffers of the 256-column table are freed
    c.params(narrow, 256)


@pytest.mark.parametrize("scene,fail_waits", [(_free_volume, False), (_free_volume, True), (_free_batch, False),
                                              (_free_batch, True), (_destroy, False), (_destroy, True),
                                              (_brick_size, False), (_wider_table, False)])
def test_no_buffer_in_use_is_handed_out(lib, scene, fail_waits):
    c = Lib(lib, fail_waits)
    before = lib.fake_violations()
    scene(c)
    assert lib.fake_violations() == before
    c.close()


def test_capture_on_another_thread_stays_valid(lib):
    """Another thread captures a stream of its own in thread-local mode, which cudaFree has no
    part in: buffers are freed, none in use is handed out, and the capture stays valid."""
    c = Lib(lib)
    before = lib.fake_violations()
    lib.fake_capture(1)
    try:
        for scene in (_free_volume, _free_batch, _destroy, _wider_table):
            scene(c)
        assert lib.fake_capture_valid()
    finally:
        lib.fake_capture(0)
    assert lib.fake_violations() == before
    c.close()


def test_everything_is_given_back(lib):
    base = lib.fake_held_bytes()
    a, b = Lib(lib), Lib(lib)
    for _ in range(3):
        for c in (a, b):
            c.ok(lib.vr_free_volume(c.h, c.open()))
            c.open(17)
    a.close()
    b.close()
    assert lib.fake_held_bytes() == base


def test_freed_memory_is_there_for_others(lib):
    """Another allocator of the process finds room for what a freed volume took, while the
    context lives."""
    c = Lib(lib)
    vid = c.open(40)
    held, used = lib.fake_held_bytes(), c.used()
    c.ok(lib.vr_free_volume(c.h, vid))
    taken = used - c.used()
    p = ctypes.c_void_p()
    lib.fake_capacity(ctypes.c_longlong(held))
    try:
        assert lib.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(taken)) == 0
    finally:
        lib.fake_capacity(ctypes.c_longlong(-1))
    lib.cudaFree(p)
    c.open(40)
    c.close()


def test_what_is_kept_is_bounded(lib):
    """A volume above the bound is given back at once; with a memory limit set, all of a volume
    is, also one opened before."""
    c = Lib(lib)
    base = lib.fake_held_bytes()
    big = c.load(320)
    c.ok(lib.vr_precompute_morphology(c.h, big, None, 0))
    assert lib.fake_held_bytes() - base > 2 << 30
    c.ok(lib.vr_free_volume(c.h, big))
    assert lib.fake_held_bytes() - base <= 2 << 30
    vid = c.load(20)
    c.ok(lib.vr_set_memory_limit(c.h, ctypes.c_ulonglong(1 << 40)))
    c.ok(lib.vr_free_volume(c.h, vid))
    assert lib.fake_held_bytes() <= base + (1 << 20)
    c.close()


def test_pool_from_the_second_study_on(lib):
    """A context that opens one study allocates as without a pool; one that opens another, and
    any beside it, from the pool, as does one that changes its derived bricks; one with a memory
    limit never."""
    before = lib.fake_pool_allocs()
    c, d = Lib(lib, reopens=False), Lib(lib, reopens=False)
    vid = c.open(20)
    c.batch(vid)
    assert lib.fake_pool_allocs() == before
    c.ok(lib.vr_free_volume(c.h, vid))
    assert lib.fake_pool_allocs() == before
    c.open(20)
    one = lib.fake_pool_allocs()
    assert one > before
    d.open(20)
    assert lib.fake_pool_allocs() > one
    e = Lib(lib, reopens=False)
    e.ok(lib.vr_set_memory_limit(e.h, ctypes.c_ulonglong(1 << 40)))
    two = lib.fake_pool_allocs()
    e.ok(lib.vr_free_volume(e.h, e.open(20)))
    e.open(20)
    assert lib.fake_pool_allocs() == two
    for x in (c, d, e):
        x.close()
    f = Lib(lib, reopens=False)  # the last context has ended: as in a new process
    vid = f.load(20)
    f.ok(lib.vr_set_brick_size(f.h, vid, 4))  # before there are derived bricks
    f.ok(lib.vr_precompute_morphology(f.h, vid, None, 0))
    assert lib.fake_pool_allocs() == two
    f.ok(lib.vr_set_brick_size(f.h, vid, 16))  # and in exchange for others
    f.ok(lib.vr_precompute_morphology(f.h, vid, None, 0))
    assert lib.fake_pool_allocs() > two
    f.close()
