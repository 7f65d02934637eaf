"""L-ORB at the sizes where its kernels' tiles and selection can go wrong, bit-exact against the
integer oracle: areas ending at, before and after the edges of the 60 x 30 tiles, the smallest image,
unaligned rows, and a periodic image whose equal responses are too many to be ranked by counting."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _same(frame, areas, points, fast_t=20, harris_t=0, tensor=None):
    import torch
    from paper_1810_03988_gb300 import LORB
    pat = synth.brief_pattern(3)
    h, w = frame.shape[:2]
    ref = oracle.lorb(frame, areas, pat, fast_t, harris_t, points)
    with LORB(w, h, points) as ctx:
        for _ in range(2):  # the second call starts from the counters that the first one left
            xy, resp, desc, cnt = ctx.detect(torch.from_numpy(frame).cuda() if tensor is None else tensor, areas, pat,
                                             fast_t, harris_t, points)
            torch.cuda.synchronize()
            n = int(cnt.cpu()[0])
            np.testing.assert_array_equal(xy[:n].cpu().numpy(), ref["xy"])
            np.testing.assert_array_equal(resp[:n].cpu().numpy(), ref["resp"])
            np.testing.assert_array_equal(desc[:n].cpu().numpy(), ref["desc"])
    return n


def _noise(w, h, seed):
    """Blocks of random colour with some noise: corners at every position relative to the tiles."""
    rng = np.random.default_rng(seed)
    img = rng.integers(0, 256, (h // 5 + 1, w // 5 + 1, 3)).repeat(5, 0).repeat(5, 1)[:h, :w]
    return np.clip(img + rng.integers(-12, 13, (h, w, 3)), 0, 255).astype(np.uint8)


@pytest.mark.parametrize("w,h", [(37, 37), (38, 40), (95, 65), (96, 66), (97, 67), (157, 128), (259, 94)])
def test_tile_edges(w, h):
    n = _same(_noise(w, h, w * h), [(0, 0, w, h)], 2048, fast_t=10)
    assert n > 0 or w < 40


@pytest.mark.parametrize("x0,y0,x1,y1", [(18, 18, 19, 19), (77, 47, 79, 50), (20, 30, 81, 61), (19, 19, 79, 49), (0, 0, 400, 20)])
def test_area_edges(x0, y0, x1, y1):
    frame = _noise(200, 150, 5)
    _same(frame, [(x0, y0, x1, y1), (x0 + 1, y0 + 1, x1 + 40, y1 + 2)], 300, fast_t=5, harris_t=-10 ** 15)


@pytest.mark.parametrize("offset,pitch", [(1, 611), (0, 613), (4, 612)])
def test_unaligned_rows(offset, pitch):
    import torch
    frame = _noise(203, 90, 9)
    buf = torch.zeros(offset + 90 * pitch, dtype=torch.uint8, device="cuda")
    t = buf[offset:].as_strided((90, 203, 3), (pitch, 3, 1))
    t.copy_(torch.from_numpy(frame))
    assert _same(frame, [(0, 0, 203, 90)], 500, tensor=t) > 0


@pytest.mark.parametrize("points", [1, 700, 2048])
def test_crowded_equal_responses(points):
    """Isolated dots on a grid: 19 000 corners of one response, ordered by their index alone."""
    frame = np.full((900, 1100, 3), 40, np.uint8)
    frame[3::7, 2::7] = 200
    assert _same(frame, [(0, 0, 1100, 900)], points) == points
