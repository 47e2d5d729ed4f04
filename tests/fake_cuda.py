"""The library's host code linked with the recording runtime of fake_cudart.c."""
import ctypes
import glob
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
HOST, DEVICE, MANAGED = 1, 2, 3


class Fake:
    def __init__(self, path):
        self.lib = ctypes.CDLL(path)
        self.lib.fake_calls.restype = ctypes.c_char_p
        self.lib.fake_mark.argtypes = [ctypes.c_void_p, ctypes.c_size_t, ctypes.c_int, ctypes.c_int]
        self.lib.lbm_last_error.restype = ctypes.c_char_p

    def clear(self):
        self.lib.fake_clear()

    def calls(self):
        return [line.split(" ") for line in self.lib.fake_calls().decode().splitlines()]

    def copies(self):
        """(destination, source, bytes) of every recorded copy."""
        return [tuple(int(v) for v in c[1:]) for c in self.calls() if c[0] == "copy"]

    def launched(self, name):
        return any(c[0] == "launch" and name in c[1] for c in self.calls())

    def waits(self):
        return sum(c[0] == "wait" for c in self.calls())

    def buffer(self, nbytes, kind, device=0):
        """A byte buffer that the runtime reports as memory of this kind."""
        b = (ctypes.c_uint8 * nbytes)()
        self.lib.fake_mark(ctypes.addressof(b), nbytes, kind, device)
        return b

    def lattice(self, nx, ny, precision=64, edges=(0, 0, 0, 0), **params):
        from paper_1601_02708_gb300._lib import Params
        p = Params(nx=nx, ny=ny, precision=precision, tau=0.8, **params)
        p.edge[:] = edges
        h = ctypes.c_void_p()
        st = self.lib.lbm_init(ctypes.byref(h), ctypes.byref(p), None, None, None, None, None, None)
        assert st == 0, self.lib.lbm_last_error()
        return h

    def state_bytes(self, h):
        n = ctypes.c_size_t()
        assert self.lib.lbm_state_bytes(h, ctypes.byref(n)) == 0
        return n.value


def load(tmp):
    from paper_1601_02708_gb300 import build
    build.build()
    objects = sorted(glob.glob(os.path.join(build.OUT_DIR, "*.o")))
    if len(objects) != len(build.sources()):
        build.build(force=True)
        objects = sorted(glob.glob(os.path.join(build.OUT_DIR, "*.o")))
    fake, lib = os.path.join(tmp, "fake_cudart.o"), os.path.join(tmp, "liblbmade_fake.so")
    subprocess.run(["gcc", "-O1", "-fPIC", "-w", "-c", os.path.join(HERE, "fake_cudart.c"), "-o", fake],
                   check=True)
    # -Bsymbolic: the recording runtime even where a real one is loaded already
    subprocess.run(["g++", "-shared", "-Wl,-Bsymbolic", "-o", lib, *objects, fake], check=True)
    return Fake(lib)
