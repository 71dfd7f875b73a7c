"""Compiles a CUDA snippet against the library's internal headers and links it with the library, for
tests of device functions and launchers that the C ABI does not reach by themselves."""
import ctypes
import os
import subprocess

from paper_2304_12597_gb300 import build as B


def compile_snippet(folder, source):
    """The snippet (namespace pd is open, pd_internal.h and pd_common.cuh included) as a ctypes library."""
    src, so = os.path.join(str(folder), "snippet.cu"), os.path.join(str(folder), "snippet.so")
    with open(src, "w") as f:
        f.write('#include "pd_internal.h"\n#include "pd_common.cuh"\nnamespace pd {\n' + source + "\n}\n")
    lib = B.build()
    cmd = [B.nvcc()] + B._flags(False) + ["-I", B.CSRC, "-shared", "-o", so, src, lib,
                                          "-Xlinker", "-rpath=" + os.path.dirname(lib)]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(so)
