"""Rigs with single-camera tiles in a kernel of their own, and rigs with many blended tiles of both kinds (at
most 2 cameras, 3 or 4), through every entry that takes them: the same canvas, bit for bit, from single calls,
the overlapped host pipeline, the batch on streams and the staged batch, which has launches of its own."""
import numpy as np
import pytest

import synth
from tests import gpu_util

pytestmark = pytest.mark.gpu


class _Camera:
    def __init__(self, width, height, x):
        self.width, self.height, self.gain = width, height, 1.0
        self.H = np.array([[1.0, 0.01, x], [-0.008, 1.0, 4.6], [1e-6, 0.0, 1.0]])


def _single_and_blended():
    cfg = synth.config_4x1080p(frames=1)
    return cfg.cameras, cfg.frame(0), cfg.canvas_w, cfg.canvas_h, cfg.levels


def _many_blended():
    """Two cameras over the whole canvas and a third over its right end."""
    cw, ch = 4400, 3000
    cams = [_Camera(cw + 8, ch + 60, -6.3), _Camera(cw - 20, ch + 60, 21.7), _Camera(700, ch + 60, cw - 500.2)]
    rng = np.random.default_rng(5)
    return cams, [rng.integers(0, 256, (c.height, c.width, 3), dtype=np.uint8) for c in cams], cw, ch, 4


@pytest.mark.parametrize("out_float", [False, True])
@pytest.mark.parametrize("scene", [_single_and_blended, _many_blended])
def test_every_entry_gives_the_same_canvas(scene, out_float):
    import torch
    from paper_1810_03988_gb300 import Batch, Rig
    cams, host, cw, ch, levels = scene()
    frames = gpu_util.gpu_frames(host)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    with Rig(cams, cw, ch, levels, out_float=out_float) as rig:
        t = rig.info()["tiles"]
        if scene is _single_and_blended:
            assert t["solo"] >= 4 * sms, t
        else:
            assert t["full4"] > 0 and t["full2"] > 0 and t["full2"] + t["full4"] >= 32 * sms, t
        ref = rig.stitch(frames).clone()
        pinned = [torch.from_numpy(f).pin_memory() for f in host]
        outs = [torch.zeros(ref.shape, dtype=ref.dtype).pin_memory() for _ in range(3)]
        for out in outs:  # consecutive calls overlap
            rig.stitch_host_async(pinned, out)
        torch.cuda.synchronize()
        for out in outs:
            assert torch.equal(out, ref.cpu())
        for mode in ("streams", "staged"):
            with pytest.MonkeyPatch.context() as mp:
                mp.setenv("STITCH_TUNE", mode)
                with Batch([rig]) as b:
                    for _ in range(2):
                        assert torch.equal(b.stitch([frames])[0], ref), mode
                    assert b.schedule()["mode"] == mode
