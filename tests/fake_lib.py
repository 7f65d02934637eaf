"""The library's host side without a GPU: its objects linked against tests/fake_cudart.cpp, whose launches,
events and copies land in a log."""
from __future__ import annotations

import collections
import ctypes
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))

Launch = collections.namedtuple("Launch", "kernel stream priority early")


class FakeLib:
    def __init__(self, directory):
        from paper_1810_03988_gb300 import _build, stitch
        _build.build()
        objs = [os.path.join(_build.BUILD, "release", os.path.basename(s)[:-3] + ".o") for s in _build._sources()]
        include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(_build.nvcc()))), "include")
        path = os.path.join(str(directory), "libstitch_fake.so")
        # -Bsymbolic: torch may have loaded the real runtime into the process
        subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", f"-I{include}", "-o", path, *objs,
                        os.path.join(HERE, "fake_cudart.cpp"), "-Wl,-Bsymbolic", "-Wl,-z,defs"], check=True)
        self.lib = ctypes.CDLL(path)
        for name, (res, args) in stitch.SIGNATURES.items():
            fn = getattr(self.lib, name)
            fn.restype, fn.argtypes = res, args
        self.lib.fake_line.restype = ctypes.c_char_p
        self.lib.fake_stream.restype = ctypes.c_void_p

    def log(self):
        """The log's lines split into words, a launch as a Launch; the log is cleared."""
        out = []
        for i in range(self.lib.fake_count()):
            w = self.lib.fake_line(i).decode().split()
            out.append(Launch(w[1], int(w[2]), int(w[3]), w[4] == "1") if w[0] == "launch" else tuple(w))
        self.lib.fake_clear()
        return out

    def rig(self, cameras, cw, ch, levels, **kw):
        from paper_1810_03988_gb300 import stitch
        desc, keep = stitch.make_desc(cameras, cw, ch, levels, **kw)
        out = ctypes.c_void_p()
        assert self.lib.stitch_rig_create(ctypes.byref(desc), 0, ctypes.byref(out)) == 0
        return out

    def frame_args(self, cameras):
        """Host frames of the cameras as pointer and pitch arrays (device memory is host memory here)."""
        n = len(cameras)
        self.frames = [ctypes.create_string_buffer(c.width * c.height * 3) for c in cameras]
        return ((ctypes.c_void_p * n)(*[ctypes.addressof(f) for f in self.frames]),
                (ctypes.c_int64 * n)(*[3 * c.width for c in cameras]))
