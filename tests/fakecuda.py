"""The library's host code without a GPU: its objects linked with a recording CUDA runtime
(fake_cudart.cpp) instead of the real one.  ``lib(folder)`` builds and loads it; ``take`` returns
the calls recorded since the last one, each as a list of words."""
import ctypes as C
import glob
import os
import subprocess

from paper_2009_09501_gb300 import build as B
from paper_2009_09501_gb300 import dibr as D

HERE = os.path.dirname(os.path.abspath(__file__))


class Fake:
    def __init__(self, folder):
        real = D.load()  # (builds the objects if they are missing or old)
        cuda = os.path.dirname(os.path.dirname(os.path.realpath(B.nvcc())))
        so = os.path.join(str(folder), "libdibr_fake.so")
        objs = [os.path.join(B.BUILD_DIR, os.path.basename(c)[:-2] + "o") for c in sorted(glob.glob(os.path.join(B.CSRC, "*.cu")))]
        if not all(os.path.exists(o) for o in objs):  # (the library without its objects)
            B.build(force=True)
        cmd = ["g++", "-std=c++17", "-O1", "-w", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I" + B.INCLUDE, "-I" + B.CSRC,
               "-I" + os.path.join(cuda, "include"), os.path.join(HERE, "fake_cudart.cpp")] + objs + ["-lpthread", "-o", so]
        r = subprocess.run(cmd, capture_output=True, text=True)
        assert r.returncode == 0, r.stderr[-3000:]
        self.lib = C.CDLL(so, mode=os.RTLD_LOCAL)
        self.lib.fake_take.restype = C.c_char_p
        for name in ("dibr_create", "dibr_destroy", "dibr_last_error", "dibr_enqueue_image", "dibr_enqueue_batch",
                     "dibr_synthesize_image", "dibr_synchronize", "dibr_set_tuning", "dibr_get_tuning", "dibr_tuning_load", "dibr_open_stream",
                     "dibr_submit_frame", "dibr_poll", "dibr_close_stream"):
            ours, theirs = getattr(self.lib, name), getattr(real, name)
            ours.restype, ours.argtypes = theirs.restype, theirs.argtypes

    def __getattr__(self, name):
        return getattr(self.lib, name)

    def take(self):
        return [line.split() for line in self.lib.fake_take().decode().splitlines()]

    def context(self):
        ctx = C.c_void_p()
        assert self.lib.dibr_create(None, C.byref(ctx)) == D.DIBR_OK
        return ctx


def image(W, H, addr=1 << 32, pitch=None):
    return D.dibr_image(addr, W, H, 3 * W if pitch is None else pitch, 1)


def outputs(names, W, first=1 << 40, pitch=None):
    """Device outputs at addresses of their own, far from one another."""
    o = D.dibr_outputs()
    for k, n in enumerate(names):
        setattr(o, n, first + (k << 34))
    o.pitch, o.depth_pitch, o.on_device = 3 * W if pitch is None else pitch, W, 1
    return o
