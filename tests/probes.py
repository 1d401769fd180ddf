"""Compiles a probe (a .cu file beside the tests that drives the library's own functions) against the built library."""
import ctypes
import os
import subprocess


def load(lib, source, directory):
    from paper_2204_03575_gb300 import build
    here, out = os.path.dirname(os.path.abspath(__file__)), os.path.join(str(directory), source + ".so")
    cmd = [build.nvcc(), *build.ARCH, *build.FLAGS, "-shared", "-o", out, os.path.join(here, source),
           lib.LIB_PATH, "-Xlinker", "-rpath", "-Xlinker", os.path.dirname(lib.LIB_PATH)]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    lib.lib()
    return ctypes.CDLL(out)
