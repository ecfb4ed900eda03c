"""Builds tests/device/kernels.cu against the library and loads it (GPU tests of single kernels)."""
import ctypes
import functools
import os
import subprocess
import tempfile

from paper_1208_6387_gb300 import _build

HERE = os.path.dirname(os.path.abspath(__file__))


def compile_kernels(out):
    _build.build()
    subprocess.run([_build.nvcc(), *_build.ARCH, *_build.FLAGS, "-shared", "-cudart", "static", "-I", _build.CSRC,
                    os.path.join(HERE, "device", "kernels.cu"), "-o", out, _build.LIB,
                    "-Xlinker", "-rpath=" + _build.OUT_DIR], check=True)
    return out


@functools.lru_cache(maxsize=1)
def load():
    tmp = tempfile.TemporaryDirectory()
    lib = ctypes.CDLL(compile_kernels(os.path.join(tmp.name, "kernels.so")))
    lib.tmp = tmp   # removed with the library
    return lib
