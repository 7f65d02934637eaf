"""The last pyramid level is formed by the tiles of the level before it: single-rig launches against the
batched staged schedule, which launches every level by itself, bit for bit, and against the oracle.
Odd canvases whose last level is smaller than a tile's halo or larger than a tile, both band precisions,
more cameras over a tile than it takes at once."""

import numpy as np
import pytest

import oracle
from tests import gpu_util

pytestmark = pytest.mark.gpu


class _Camera:
    def __init__(self, width, height, H):
        self.width, self.height, self.H, self.gain = width, height, H, 1.0


@pytest.mark.parametrize("fp16", [False, True])
@pytest.mark.parametrize("cams,levels,cw,ch", [(2, 3, 301, 203), (2, 4, 301, 203), (5, 4, 997, 301), (6, 6, 1203, 331),
                                               (3, 7, 517, 229)])
def test_last_level_inside_the_one_before(cams, levels, cw, ch, fp16, monkeypatch):
    import torch
    from paper_1810_03988_gb300 import Batch, Rig
    w, h = max(160, int(2.2 * cw / cams)), int(ch * 0.95)
    cs = [_Camera(w, h, np.array([[1.0, 0.01, (cw - w) * i / (cams - 1) + 0.3], [-0.008, 1.0, 4.6], [1e-6, 0.0, 1.0]]))
          for i in range(cams)]
    rng = np.random.default_rng(cams * 100 + levels)
    frames = [rng.integers(0, 256, (h, w, 3), dtype=np.uint8) for _ in cs]
    dev = gpu_util.gpu_frames(frames)
    monkeypatch.setenv("STITCH_TUNE", "staged")
    with Rig(cs, cw, ch, levels, band_fp16=fp16, out_float=True) as rig:
        got = rig.stitch(dev)
        with Batch([rig]) as b:
            assert torch.equal(b.stitch([dev])[0], got)
        got = got.cpu().numpy()
    ref = oracle.forward(cs, frames, cw, ch, levels)
    gpu_util.compare(got, ref, True, gpu_util.TOL_F16 if fp16 else gpu_util.TOL_F32)
