"""What the library's host side hands the GPU, call by call, on a CUDA runtime that only takes notes."""
import ctypes
import re
import struct

import numpy as np
import pytest

import synth
from tests.fake_lib import FakeLib, Launch


class _Camera:
    def __init__(self, width, height, H, gain=1.0):
        self.width, self.height, self.H, self.gain = width, height, H, gain


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    return FakeLib(tmp_path_factory.mktemp("fake"))


def _shift(x, y):
    return np.array([[1.0, 0.0, x], [0.0, 1.0, y], [0.0, 0.0, 1.0]])


def _apart():
    """Two cameras far apart: solo canvas tiles (more than 4 per SM) and empty ones between, nothing blended."""
    return [_Camera(1600, 1400, _shift(-20.0, -20.0)), _Camera(1600, 1400, _shift(2200.0, -20.0))], 3776, 1344


def _two():
    cfg = synth.config_2cam(scale=0.25)
    return cfg.cameras, cfg.canvas_w, cfg.canvas_h


def _stitch(fake, rig, cams, cw, ch, entry="stitch_frames", stream=None, elem=3):
    fp, pt = fake.frame_args(cams)
    out = ctypes.create_string_buffer(cw * ch * elem)
    fake.log()
    assert getattr(fake.lib, entry)(rig, fp, pt, out, cw * elem, stream) == 0
    return fake.log()


def _first_after_waits(log):
    """Per stream, the launches whose predecessor on the stream is an event wait."""
    last, out = {}, []
    for e in log:
        if isinstance(e, Launch):
            if last.get(e.stream) == "wait":
                out.append(e)
            last[e.stream] = "launch"
        elif e[0] == "wait":
            last[int(e[1])] = "wait"
    return out


@pytest.mark.parametrize("entry", ["stitch_frames", "stitch_frames_host_async", "batch"])
@pytest.mark.parametrize("path", ["fused", "plain"])
@pytest.mark.parametrize("scene", [_apart, _two])
def test_no_launch_that_follows_an_event_wait_is_programmatic(fake, entry, path, scene, monkeypatch):
    if path == "plain" and entry == "batch":
        pytest.skip("a batch takes fused rigs")
    cams, cw, ch = scene()
    rig = fake.rig(cams, cw, ch, 3, path=path)
    if entry == "batch":
        monkeypatch.setenv("STITCH_TUNE", "streams")
        batch = ctypes.c_void_p()
        assert fake.lib.stitch_batch_create((ctypes.c_void_p * 1)(rig), 1, ctypes.byref(batch)) == 0
        fp, pt = fake.frame_args(cams)
        out = ctypes.create_string_buffer(cw * ch * 3)
        args = ((ctypes.c_void_p * 1)(ctypes.addressof(fp)), (ctypes.c_void_p * 1)(ctypes.addressof(pt)),
                (ctypes.c_void_p * 1)(ctypes.addressof(out)), (ctypes.c_int64 * 1)(3 * cw))
        for _ in range(2):  # the first call times the schedules
            fake.log()
            assert fake.lib.stitch_batch_frames(batch, *args, None) == 0
        log = fake.log()
        fake.lib.stitch_batch_destroy(batch)
    else:
        log = _stitch(fake, rig, cams, cw, ch, entry)
    launches = [e for e in log if isinstance(e, Launch)]
    assert any("k_solo" in e.kernel for e in launches) == (scene is _apart and path == "fused")
    after = _first_after_waits(log)
    assert (len(after) > 0) == (entry != "stitch_frames")
    assert not [e for e in after if e.early], after
    # the launches behind them overlap, and so does the first one on the caller's stream
    chain = [e for e in launches if "k_solo" not in e.kernel and e not in after]
    assert all(e.early for e in chain), chain
    fake.lib.stitch_rig_destroy(rig)


@pytest.mark.parametrize("priority", [0, -3])
@pytest.mark.parametrize("scene", [_apart, _two])
def test_a_call_runs_on_the_caller_s_stream_at_its_priority(fake, scene, priority):
    cams, cw, ch = scene()
    streams = fake.lib.fake_streams()
    rig = fake.rig(cams, cw, ch, 3)
    assert fake.lib.fake_streams() == streams, "a rig has no stream of its own"
    stream = fake.lib.fake_stream(priority)
    launches = [e for e in _stitch(fake, rig, cams, cw, ch, stream=stream) if isinstance(e, Launch)]
    assert len(launches) > 3
    assert len({e.stream for e in launches}) == 1 and {e.priority for e in launches} == {priority}, launches
    fake.lib.stitch_rig_destroy(rig)


def test_lorb_counts_are_cleared_after_a_refused_launch(fake):
    """The counters of a detection are cleared by its own kernels; a sequence that a refused launch cuts
    short leaves that to the next call."""
    from paper_1810_03988_gb300 import stitch
    W, H, N = 64, 64, 8
    ctx = ctypes.c_void_p()
    assert fake.lib.stitch_lorb_create(W, H, N, 0, ctypes.byref(ctx)) == 0
    frame, out = ctypes.create_string_buffer(3 * W * H), [ctypes.create_string_buffer(64 * N) for _ in range(4)]
    areas, pattern = (ctypes.c_int32 * 4)(0, 0, W, H), (ctypes.c_int8 * 1024)()

    def detect():
        fake.log()
        st = fake.lib.stitch_lorb_detect(ctx, frame, W, H, 3 * W, areas, 1, ctypes.byref(stitch.stitch_lorb_params(20, 0, N)),
                                         pattern, *out, None)
        log = fake.log()
        return st, [e[2] for e in log if e[0] == "memset"], [e.kernel for e in log if isinstance(e, Launch)]

    st, cleared, kernels = detect()
    assert st == 0 and not cleared and len(kernels) == 3
    for refused in (1, 2):  # behind lorb_detect, behind lorb_prune
        fake.lib.fake_refuse(refused)
        st, cleared, kernels = detect()
        assert st == stitch.STITCH_ECUDA and not cleared and len(kernels) == 2
        st, cleared, kernels = detect()
        assert st == 0 and len(kernels) == 3
        assert len(cleared) == 1 and int(cleared[0]) >= 4 * (4 + 1024), "the counters and the histogram"
        st, cleared, _ = detect()
        assert st == 0 and not cleared
    fake.lib.stitch_lorb_destroy(ctx)


def test_schedules_timed_with_earlier_kernels_are_timed_again(fake, monkeypatch, tmp_path):
    """The tuning cache's key changes with the kernels that the tuner times: a line stored by a library with
    earlier ones (key version 2) is not taken, a line stored by this one is."""
    cams, cw, ch = _two()
    rig = fake.rig(cams, cw, ch, 3)
    blob = b"libstitch batch schedule %d\0" + struct.pack("<i", 1)
    blob += struct.pack("<9i", len(cams), cw, ch, 3, 0, 0, 0, 0, 0) + struct.pack("<3d", 0.0, 0.0, 0.0)
    for c in cams:
        blob += struct.pack("<ii", c.width, c.height) + np.asarray(c.H, np.float64).tobytes() + struct.pack("<f", c.gain)

    def line(version, mode):
        h = 1469598103934665603
        for byte in blob % version:
            h = (h ^ byte) * 1099511628211 % 2 ** 64
        return '{"key": "fake|152|%016x", "mode": "%s", "order": 1, "variant": 1, "chunk": 4, "shape": 0, "ms": 1.0}\n' % (h, mode)

    cache = tmp_path / "tune"
    monkeypatch.setenv("STITCH_TUNE_CACHE", str(cache))
    monkeypatch.delenv("STITCH_TUNE", raising=False)

    def from_cache():
        batch = ctypes.c_void_p()
        assert fake.lib.stitch_batch_create((ctypes.c_void_p * 1)(rig), 1, ctypes.byref(batch)) == 0
        fp, pt = fake.frame_args(cams)
        out = ctypes.create_string_buffer(cw * ch * 3)
        args = ((ctypes.c_void_p * 1)(ctypes.addressof(fp)), (ctypes.c_void_p * 1)(ctypes.addressof(pt)),
                (ctypes.c_void_p * 1)(ctypes.addressof(out)), (ctypes.c_int64 * 1)(3 * cw))
        assert fake.lib.stitch_batch_frames(batch, *args, None) == 0
        order = ctypes.c_int32()
        assert fake.lib.stitch_batch_get_schedule(batch, ctypes.byref(order), None, None) == 0
        fake.lib.stitch_batch_destroy(batch)
        return bool(order.value >> 24 & 1)

    cache.write_text(line(2, "streams"))
    assert not from_cache()          # timed, and stored behind the old line
    assert len(cache.read_text().splitlines()) == 2
    assert from_cache()
    cache.write_text(line(3, "streams"))
    assert from_cache()              # the key is formed as this test forms it
    fake.lib.stitch_rig_destroy(rig)


@pytest.mark.parametrize("spread", [1.0, 1.12])  # source pixels per canvas pixel: footprints of either capacity
@pytest.mark.parametrize("cw,ch", [(1200, 400), (7000, 2000)])  # about one wave of down1 tiles, and many
def test_the_sweep_of_down1_goes_by_the_number_of_waves(fake, spread, cw, ch):
    w, h = int(0.6 * cw * spread), int(0.9 * ch * spread)
    cams = [_Camera(w, h, np.diag([1 / spread, 1 / spread, 1.0]) + _shift(x, 0.05 * ch) - np.eye(3)) for x in (0.0, 0.4 * cw)]
    rig = fake.rig(cams, cw, ch, 3)
    log = _stitch(fake, rig, cams, cw, ch)
    down1 = [e.kernel for e in log if isinstance(e, Launch) and "k_down1" in e.kernel]
    assert len(down1) == 1
    capacity, rolled = re.search(r"k_down1I6float4Li(\d+)ELb([01])E", down1[0]).groups()
    assert int(capacity) == (1536 if spread == 1.0 else 2048)
    assert rolled == ("1" if cw == 7000 else "0")
    fake.lib.stitch_rig_destroy(rig)
