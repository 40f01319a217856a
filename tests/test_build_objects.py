"""The built objects hold their device code uncompressed: a process's first launch from a
compressed one waits for its decompression (11 ms for the backward's kernels)."""

import glob
import os

from paper_2605_19737_gb300 import build as native


def test_device_code_is_not_compressed():
    native.build(debug=False)
    objects = sorted(glob.glob(os.path.join(native.BUILD, "*.o")))
    assert {os.path.basename(s)[:-3] for s in native.sources()} == {os.path.basename(o)[:-2] for o in objects}
    for o in objects:
        with open(o, "rb") as f:
            data = f.read()
        host_only = b".nv_fatbin" not in data
        # the object's own ELF header, and that of the device code inside
        assert host_only or data.count(b"\x7fELF") >= 2, os.path.basename(o)
