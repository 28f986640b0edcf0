"""Compiles a CUDA source that includes the library's own into a shared object for ctypes."""
import ctypes
import os
import subprocess

PKG = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1807_01151_gb300")


def compile_cuda(source, folder, link_library=False):
    from paper_1807_01151_gb300 import build
    src, lib = os.path.join(folder, "unit.cu"), os.path.join(folder, "unit.so")
    with open(src, "w") as f:
        f.write(source)
    extra = [build.LIB, "-Xlinker", "-rpath," + PKG] if link_library else []
    cmd = [build.NVCC] + build.ARCH + build.FLAGS + ["-I", build.CSRC, "-shared", src, "-o", lib] + extra
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(lib)
