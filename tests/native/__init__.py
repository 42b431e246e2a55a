"""Small CUDA libraries of the tests: each .cu here is compiled against the package's
sources and libnne.so, for tests of device functions and launchers behind the C ABI."""
import ctypes
import os
import subprocess

from paper_2501_13237_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


def library(name):
    build.build()
    src, out = os.path.join(HERE, name + ".cu"), os.path.join(build.BUILD, f"test_{name}.so")
    newest = max(os.path.getmtime(p) for p in [src, build.LIB] + build._headers())
    if not os.path.exists(out) or os.path.getmtime(out) < newest:
        cmd = [build.nvcc(), *build.ARCH, *build.FLAGS, "-I", build.CSRC, "-shared", src, "-o", out, build.LIB, "-lcudart",
               "-Xlinker", "-rpath", "-Xlinker", build.PKG]
        r = subprocess.run(cmd, capture_output=True, text=True)
        assert r.returncode == 0, r.stderr[-4000:]
    return ctypes.CDLL(out)
