"""Access to the library's internal state for tests: a small shared object compiled from a source string
with the library's own headers and linked to libmh.so."""
import ctypes
import os
import subprocess
import tempfile

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_1007_5335_gb300")
NVCC = "/usr/local/cuda/bin/nvcc"


def compile_cuda(source: str, link_lib: bool = True) -> ctypes.CDLL:
    """CDLL of a CUDA source string."""
    with tempfile.TemporaryDirectory() as d:
        src, out = os.path.join(d, "access.cu"), os.path.join(d, "access.so")
        with open(src, "w") as f:
            f.write(source)
        cmd = [NVCC, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O2", "-shared", "-Xcompiler", "-fPIC",
               "-I", os.path.join(PKG, "csrc"), "-I", os.path.join(ROOT, "include"), src, "-o", out]
        if link_lib:
            cmd += [os.path.join(PKG, "libmh.so"), "-Xlinker", "-rpath=" + PKG]
        r = subprocess.run(cmd, capture_output=True, text=True)
        assert r.returncode == 0, r.stderr
        return ctypes.CDLL(out)
