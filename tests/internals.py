"""Builds and loads tests/native/internals.cu: the library's internals for tests that
plant mistakes or reach functions that the C ABI does not export."""
import ctypes
import os
import subprocess

from paper_1901_10026_gb300 import build as tgbuild

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(HERE, "native", "internals.cu")
LIB = os.path.join(HERE, "native", "internals.so")
_lib = None


def load() -> ctypes.CDLL:
    """The test library, compiled when it is older than its source or libtg.so."""
    global _lib
    if _lib is None:
        tg = tgbuild.build()
        if not os.path.exists(LIB) or os.path.getmtime(LIB) < max(os.path.getmtime(SRC), os.path.getmtime(tg)):
            tmp = LIB + f".tmp{os.getpid()}"
            subprocess.check_call([tgbuild.nvcc(), *tgbuild.ARCH, *tgbuild.FLAGS, "-I", tgbuild.CSRC, "-shared",
                                   "-o", tmp, SRC, tg, "-Xlinker", "-rpath=" + os.path.dirname(tg)])
            os.replace(tmp, LIB)
        _lib = ctypes.CDLL(LIB)
    return _lib
