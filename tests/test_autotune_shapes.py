"""Which launches the autotuner times: launch shapes only where the render uses them."""

import numpy as np
import pytest
import torch

from paper_2605_19737_gb300 import autotune


class _Context:
    device = 0

    def __init__(self):
        self.shapes = []

    def render(self, vol, cams, W, H, out, kernel, packet_w, warps_per_block):
        self.shapes.append((packet_w, warps_per_block))


@pytest.mark.parametrize("W,H,n,shapes", [(128, 128, 1, 1), (500, 400, 1, 1), (501, 400, 1, 9), (128, 128, 12, 1),
                                          (128, 128, 13, 9), (60, 60, 100, 9), (50, 50, 200, 1), (1920, 1080, 1, 9)])
def test_candidates(monkeypatch, tmp_path, W, H, n, shapes):
    monkeypatch.setattr(torch.cuda, "get_device_name", lambda d: "none")
    monkeypatch.setattr(autotune, "_time", lambda launch, reps: launch() or 1.0)
    ctx = _Context()
    kw = dict(out=object(), cache_path=str(tmp_path / "c.json"), prepare=lambda cells: None)
    t = autotune.tune_render(ctx, 1, np.zeros((n, 12)), W, H, "k", **kw)
    assert len(set(ctx.shapes)) == shapes and len(t["timings"]) == 3 * shapes
    assert shapes > 1 or (t["packet_w"], t["warps_per_block"]) == (4, 4)
    # shapes that are asked for are timed
    ctx = _Context()
    t = autotune.tune_render(ctx, 1, np.zeros((n, 12)), W, H, "j", candidates=[(8, 2), (16, 4)], **kw)
    assert set(ctx.shapes) == {(8, 2), (16, 4)}
