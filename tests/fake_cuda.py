"""The library's host code on a CUDA runtime without a GPU (fake_cudart.cpp)."""
import ctypes
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))


class Fake:
    """``lib``: the C ABI over the fake runtime; the methods steer and read it."""

    def __init__(self, lib):
        self.lib = lib
        lib.fake_log.restype = ctypes.c_char_p
        lib.fake_reset.argtypes = [ctypes.c_size_t]
        lib.fake_used.restype = ctypes.c_size_t

    def reset(self, limit=0):
        self.lib.fake_reset(limit)

    def log(self):
        return self.lib.fake_log().decode().splitlines()

    def launches(self):
        return [x.split()[1] for x in self.log() if x.startswith("launch")]

    def used(self):
        return self.lib.fake_used()

    def host_mapped(self, on=True):
        self.lib.fake_host_mapped(int(on))

    def capturing(self, on=True):
        self.lib.fake_capturing(int(on))

    def elapsed(self, ms):
        self.lib.fake_elapsed((ctypes.c_float * len(ms))(*ms), len(ms))


def load(folder):
    """Links the library's objects with the fake runtime (all calls bound inside)
    and loads the result through the package's own binding."""
    from paper_2602_13385_gb300 import _lib, build
    build.build()
    objs = [os.path.join(build.OBJ, s.replace(".cu", ".o")) for s in build.SOURCES]
    if not all(os.path.exists(o) for o in objs):
        build.build(force=True)
    so = os.path.join(str(folder), "libscf_fake.so")
    inc = os.path.join(os.path.dirname(os.path.dirname(build.nvcc())), "include")
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-Wl,-Bsymbolic", "-I", inc, "-o", so,
                    os.path.join(HERE, "fake_cudart.cpp"), *objs], check=True)
    real, path = _lib._lib, build.LIB
    try:
        _lib._lib, build.LIB = None, so
        return Fake(_lib.load(build=False))
    finally:
        _lib._lib, build.LIB = real, path
