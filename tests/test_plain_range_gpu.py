"""The plain path where a collapsed level leaves the range of single precision: an infinite sample reaches the
pixels whose EXPAND has a tap on it, and no others.  (An odd position has the taps k and k + 1 only; a third one
of weight 0 would turn an infinite neighbour into a NaN.)"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

W, H, CW, STEP, LEVELS = 64, 64, 96, 32, 3


def _fold(i, n):
    i = np.abs(i)
    return np.where(i < n, i, 2 * (n - 1) - i)


def _reduce(a):
    for axis in (0, 1):
        n = a.shape[axis]
        at = 2 * np.arange((n + 1) // 2)
        a = sum(w / 16 * np.take(a, _fold(at + k, n), axis) for k, w in zip(range(-2, 3), (1, 4, 6, 4, 1)))
    return a


def _taps(x):
    return [(x // 2 + k, w) for k, w in ((-1, 0.125), (0, 0.75), (1, 0.125))] if x % 2 == 0 else [(x // 2, 0.5), (x // 2 + 1, 0.5)]


def _expand(a, shape):
    for axis in (0, 1):
        n = a.shape[axis]
        a = np.stack([sum(w * np.take(a, int(_fold(np.array(k), n)), axis) for k, w in _taps(x)) for x in range(shape[axis])], axis)
    return a


def _collapsed(images, weights):
    """R^0, R^1 and R^2 of the blend in 64 bits."""
    g, a = [[i] for i in images], [[w] for w in weights]
    for p in g + a:
        for _ in range(LEVELS - 1):
            p.append(_reduce(p[-1]))
    r = [None] * LEVELS
    for l in range(LEVELS - 1, -1, -1):
        top = l == LEVELS - 1
        band = [p[l] if top else p[l] - _expand(p[l + 1], p[l].shape) for p in g]
        den = sum(p[l] for p in a)
        r[l] = sum(p[l] * b for p, b in zip(a, band)) / np.maximum(den, 1e-12) + (0.0 if top else _expand(r[l + 1], g[0][l].shape))
    return r


@pytest.mark.parametrize("seed", [2, 4, 9])
def test_an_infinite_sample_stays_within_its_taps(seed):
    import torch
    from paper_1810_03988_gb300 import Rig

    class Camera:  # an image seen at a whole number of pixels: samples are texels
        width, height, gain = W, H, float(np.finfo(np.float32).max)

        def __init__(self, x):
            self.H = np.array([[1.0, 0.0, x], [0.0, 1.0, 0.0], [0.0, 0.0, 1.0]])

    rng = np.random.default_rng(seed)
    views = [np.kron(rng.integers(0, 2, (H // 8, W // 8)), np.ones((8, 8))) for _ in range(2)]  # black and white blocks
    frames = [np.repeat((255 * v).astype(np.uint8)[:, :, None], 3, 2) for v in views]
    # the cameras' images on the canvas (clamped outside) and the seam between them, in units of the largest float
    x = np.arange(CW)
    images = [v[:, np.clip(x - s, 0, W - 1)] for v, s in zip(views, (0, STEP))]
    y = np.minimum(np.arange(H), H - 1 - np.arange(H))[:, None] + 0.5
    wa = np.minimum(np.minimum(x, W - 1 - x) + 0.5, y)
    wb = np.minimum(np.minimum(x - STEP, W - 1 - (x - STEP)) + 0.5, y)
    first = (wa > 0) & (wa >= wb)
    r0, r1, r2 = _collapsed(images, [first.astype(float), 1.0 - first])
    over, fits = np.abs(r1) > 1.01, np.abs(r1) < 0.99
    for j, i in np.argwhere(fits):  # nor may a sample of the last level that it takes have rounded up to infinity
        fits[j, i] = all(abs(r2[_fold(np.array(b), len(r2)), _fold(np.array(a), r2.shape[1])]) < 0.99
                         for b, _ in _taps(j) for a, _ in _taps(i))
    expect, beside = [], 0
    for py in range(8, H - 8):
        for px in range(8, CW - 8):
            ty, tx = [k for k, _ in _taps(py)], [k for k, _ in _taps(px)]
            if abs(r0[py, px]) < 0.01 or not all(fits[j, i] for j in ty for i in tx):
                continue
            expect.append((py, px, 1.0 if r0[py, px] > 0 else 0.0))
            near = [(j, i) for j in {ty[0] - (py % 2), *ty} for i in {tx[0] - (px % 2), *tx}]
            beside += r0[py, px] > 0 and any(over[j, i] for j, i in near)
    assert beside > 0, "some pixel has an infinite sample next to its taps"
    with Rig([Camera(0), Camera(STEP)], CW, H, LEVELS, out_float=True, path="plain", weights="seam") as rig:
        got = rig.stitch([torch.from_numpy(f).cuda() for f in frames]).cpu().numpy()
    for py, px, v in expect:
        assert (got[py, px] == v).all(), (py, px, got[py, px], v)
