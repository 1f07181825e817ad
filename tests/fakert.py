"""The library's host side over a CUDA runtime without a device
(fake_cudart.cpp): built once per session, called through the package's own
bindings.  Every kernel does nothing, so counts and flags come out zero."""
import contextlib
import ctypes
import glob
import os
import subprocess
import tempfile

import paper_2507_06579_gb300 as E
from paper_2507_06579_gb300 import _build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
_fake = None


def load():
    """ctypes handle of the library linked with the fake runtime."""
    global _fake
    if _fake is None:
        E.build()
        objs = sorted(glob.glob(os.path.join(_build.BUILD, "*.cu.o")))
        if len(objs) < len(_build.sources()):  # the library without its objects
            E.build(force=True)
            objs = sorted(glob.glob(os.path.join(_build.BUILD, "*.cu.o")))
        inc = os.path.join(os.path.dirname(os.path.dirname(_build.nvcc())), "include")
        out = os.path.join(tempfile.mkdtemp(), "libeis_fake.so")
        subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", inc,
                        os.path.join(ROOT, "tests", "fake_cudart.cpp"),
                        *objs,
                        "-o", out, "-ldl", "-lpthread"], check=True)
        L = ctypes.CDLL(out)
        for name, res, args in E.SIGNATURES:
            f = getattr(L, name)
            f.restype, f.argtypes = res, args
        L.fake_launches.argtypes = [ctypes.c_char_p]
        L.fake_launches.restype = L.fake_violations.restype = L.fake_waits.restype = ctypes.c_long
        L.fake_mapped.restype = L.fake_peak.restype = ctypes.c_ulonglong
        L.fake_set_capacity.argtypes = [ctypes.c_ulonglong]
        L.fake_fail_after.argtypes = [ctypes.c_long, ctypes.c_long]
        L.fake_capture.argtypes = [ctypes.c_void_p, ctypes.c_int]
        _fake = L
    return _fake


@contextlib.contextmanager
def installed():
    """The package calls the fake library inside the block (the block yields it)."""
    L, saved = load(), E._lib
    E._lib = L
    L.fake_set_capacity(200 << 30)
    L.fake_reset()
    try:
        yield L
    finally:
        L.fake_fail_after(-1, 0)
        L.fake_set_capacity(200 << 30)
        E._lib = saved
