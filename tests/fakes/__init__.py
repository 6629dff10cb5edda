"""The library linked against a CUDA runtime that needs no GPU (cudart.cpp)."""
import contextlib
import ctypes
import gc
import importlib
import os
import subprocess

from paper_2607_11951_gb300 import grid as G

B = importlib.import_module("paper_2607_11951_gb300.build")  # (the package has a function of this name)
DEFAULT_SMEM = 48 * 1024  # shared memory of a block, its own and dynamic, without an attribute
HERE = os.path.dirname(os.path.abspath(__file__))


def link(folder):
    """libgrid's objects and the stand-in as one library in `folder`."""
    objs = [os.path.join(B.OUT, s + ".o") for s in B.SOURCES]
    if not all(map(os.path.exists, objs)):
        B.build()
    out = os.path.join(str(folder), "libgrid_fake.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-Wl,-Bsymbolic", os.path.join(HERE, "cudart.cpp")]
                   + objs + ["-o", out], check=True)
    return out


class Runtime:
    def __init__(self, path):
        self.L = ctypes.CDLL(path)
        self.L.fake_launches.restype = ctypes.c_char_p

    def reset(self, fail_at=0, ones=0):
        self.L.fake_reset(ctypes.c_long(fail_at), ctypes.c_long(ones))

    def get(self, name):
        return ctypes.c_long.in_dll(self.L, "fake_" + name).value

    def launches(self):
        """(kernel, grid, threads, dynamic shared memory, its limit) per launch since the last reset."""
        out = []
        for line in self.L.fake_launches().decode().splitlines():
            name, *x = line.split()
            x = list(map(int, x))
            out.append((name, tuple(x[:3]), x[3], x[4], x[5]))
        return out


@contextlib.contextmanager
def use(path):
    """The binding on the library at `path`; objects made inside are freed inside."""
    gc.collect()
    was = G.library_path, G._lib, G._stream
    G.library_path, G._lib, G._stream = (lambda: path), None, (lambda stream: ctypes.c_void_p(0))
    try:
        yield Runtime(path)
    finally:
        gc.collect()
        G.library_path, G._lib, G._stream = was
