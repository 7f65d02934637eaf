"""Canvas tiles that one camera alone fills and under which no pyramid level is read: they are warped
by a kernel of their own beside the pyramid's launches.  Odd canvas sizes (partial tiles at the right and
bottom border), 8-bit rows with and without word alignment, float output, both canvas models, a rig whose
other tiles are blended, and a call captured in a CUDA graph."""
import numpy as np
import pytest

import oracle
import synth
from tests import gpu_util

pytestmark = pytest.mark.gpu


class _Camera:
    def __init__(self, width, height, H, gain):
        self.width, self.height, self.H, self.gain = width, height, H, gain


def _one_camera(cyl):
    """One camera that fills an odd-sized canvas of more than 4 tiles per SM: (camera, size, canvas)."""
    if cyl:
        K = np.array([[700.0, 0.0, 700.3], [0.0, 700.0, 600.1], [0.0, 0.0, 1.0]])
        return _Camera(1400, 1200, K, 1.0), (1473, 1201), (1000.0, 736.0, 600.0)
    M = np.array([[1.05, 0.02, -41.3], [-0.015, 1.04, -23.7], [1e-6, -2e-6, 1.0]])
    return _Camera(1999, 1501, M, 0.9), (1967, 1459), None


@pytest.mark.parametrize("cyl", [False, True])
@pytest.mark.parametrize("output", ["u8", "u8_unaligned", "f32"])
def test_single_camera_canvas(cyl, output):
    import torch
    from paper_1810_03988_gb300 import Rig
    cam, (cw, ch), canvas = _one_camera(cyl)
    frame = np.random.default_rng(3).integers(0, 256, (cam.height, cam.width, 3), dtype=np.uint8)
    is_float = output == "f32"
    ref = oracle.forward([cam], [frame], cw, ch, 3, canvas=canvas)
    with Rig([cam], cw, ch, 3, out_float=is_float, canvas=canvas) as rig:
        t = rig.info()["tiles"]
        assert t["solo"] == ((cw + 63) // 64) * ((ch + 31) // 32), t
        if output == "u8":  # rows of whole words
            out = torch.zeros((ch, (cw + 3) // 4 * 4, 3), dtype=torch.uint8, device="cuda")[:, :cw]
        else:
            out = torch.zeros((ch, cw, 3), dtype=torch.float32 if is_float else torch.uint8, device="cuda")
        got = rig.stitch(gpu_util.gpu_frames([frame]), out).cpu().numpy()
    gpu_util.compare(got, ref, is_float)


def test_beside_the_pyramid_and_captured():
    """Full-size 4 x 1080p: the same canvas eagerly, from a second stream and from a replayed graph, and
    the same as the batched schedules, which send every tile through the pyramid's kernel."""
    import torch
    from paper_1810_03988_gb300 import Batch, Rig
    cfg = synth.config_4x1080p(frames=1)
    frames = gpu_util.gpu_frames(cfg.frame(0))
    with Rig(cfg.cameras, cfg.canvas_w, cfg.canvas_h, cfg.levels) as rig:
        ref = rig.stitch(frames).clone()
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        out = torch.zeros_like(ref)
        with torch.cuda.stream(side):
            rig.stitch(frames, out)
        side.synchronize()
        assert torch.equal(out, ref)
        out.zero_()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            rig.stitch(frames, out)
        for _ in range(2):
            out.zero_()
            graph.replay()
            torch.cuda.synchronize()
            assert torch.equal(out, ref)
        with pytest.MonkeyPatch.context() as mp:
            mp.setenv("STITCH_TUNE", "staged")
            with Batch([rig]) as b:
                got = b.stitch([frames])[0]
        assert torch.equal(got, ref)
