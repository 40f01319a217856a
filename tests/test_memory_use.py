"""Under a memory limit everything fits that fits without the skip fields, which are optional:
they are left out, or given up when another buffer needs their room. On a CUDA runtime without a
GPU (tests/native/fake_cuda.cpp)."""

import ctypes

import numpy as np
import pytest

from tests.test_freed_buffers import Lib, lib  # noqa: F401

DIMS = 50


class Cycle(Lib):
    """Two volumes opened, rendered, differentiated, filtered and batched in one context."""

    def derived(self, vid):
        n, a, b = ctypes.c_longlong(), ctypes.c_ulonglong(), ctypes.c_ulonglong()
        self.ok(self.lib.vr_get_layout(self.h, vid, ctypes.byref(n), ctypes.byref(a), ctypes.byref(b)))
        return b.value

    def render(self, vid):
        img = np.zeros((8, 8, 4), np.float32)
        cam = (ctypes.c_float * 12)()
        self.ok(self.lib.vr_render(self.h, vid, cam, 1, 8, 8, ctypes.c_void_p(img.ctypes.data), 0, None, None, None))

    def run(self):
        lib, h = self.lib, self.h
        sig = (ctypes.c_float * 1)(1.0)
        vids = []
        for _ in range(2):
            vid = self.load(DIMS)
            self.ok(lib.vr_precompute_morphology(h, vid, sig, 1))
            self.params(vid, 4096)
            self.render(vid)
            vids.append(vid)
        bid = self.batch(vids[0], 40)
        img = np.zeros((8, 8, 4), np.float32)
        cam, dtf = (ctypes.c_float * 12)(), np.zeros((1, 4096, 4), np.float32)
        dvol = np.zeros((DIMS,) * 3, np.float32)
        for vid in vids:
            self.ok(lib.vr_render_backward(h, vid, cam, 1, 8, 8, ctypes.c_void_p(img.ctypes.data),
                                           ctypes.c_void_p(dtf.ctypes.data), None, ctypes.c_void_p(dvol.ctypes.data),
                                           None))
            self.ok(lib.vr_prefilter(h, vid, 1, ctypes.c_float(1.0)))
            self.ok(lib.vr_precompute_morphology(h, vid, sig, 1))
            self.render(vid)
            assert self.derived(vid) > 0
        self.ok(lib.vr_batch_update(h, bid))
        self.ok(lib.vr_batch_render(h, bid, None, None))
        return self.used()


def _without_fields(lib):
    """The use of a cycle whose volumes get no field: the allocation of each is made to fail."""
    c = Cycle(lib, reopens=False)
    sig = (ctypes.c_float * 1)(1.0)
    for _ in range(2):
        vid = c.load(DIMS)
        c.ok(lib.vr_debug_fail_alloc(c.h, ctypes.c_longlong(1), None))  # the derived bricks, then the cell ranges
        c.ok(lib.vr_precompute_morphology(c.h, vid, None, 0))
        assert c.derived(vid) > 0
    lean = c.used()
    c.close()
    full = Cycle(lib, reopens=False)
    for _ in range(2):
        vid = full.load(DIMS)
        full.ok(lib.vr_precompute_morphology(full.h, vid, None, 0))
    fields = full.used() - lean
    full.close()
    return fields


@pytest.mark.parametrize("more", [0, 1000, 100000, 10 ** 9])
def test_a_limit_without_room_for_fields(lib, more):  # noqa: F811
    c = Cycle(lib, reopens=False)
    use = c.run()
    c.close()
    fields = _without_fields(lib)
    cells = (DIMS - 1) ** 3
    assert fields > 2 * 5 * cells
    before = lib.fake_violations()
    c = Cycle(lib, reopens=False)
    c.ok(lib.vr_set_memory_limit(c.h, ctypes.c_ulonglong(use - fields + more)))
    assert c.run() <= use - fields + more
    assert lib.fake_violations() == before
    c.close()


def test_a_full_device(lib):  # noqa: F811
    """The same without a limit, on a device with room for the buffers but not for the fields."""
    c = Cycle(lib, reopens=False)
    base = lib.fake_held_bytes()
    c.run()
    use = lib.fake_held_bytes() - base
    c.close()
    fields = _without_fields(lib)
    c = Cycle(lib, reopens=False)
    lib.fake_capacity(ctypes.c_longlong(lib.fake_held_bytes() + use - fields + 4096))
    try:
        c.run()
    finally:
        lib.fake_capacity(ctypes.c_longlong(-1))
    c.close()
