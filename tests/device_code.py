"""Compiles a test's own launchers of the library's device functions (csrc headers) with nvcc."""
import ctypes
import os
import subprocess

from paper_2112_05051_gb300 import build


def compile_device(source, folder, link=()):
    """ctypes library of the CUDA source text, built in `folder`; `link`: libraries it calls."""
    src, out = os.path.join(str(folder), "t.cu"), os.path.join(str(folder), "libt.so")
    with open(src, "w") as f:
        f.write(source)
    subprocess.run([build.nvcc(), "-shared", "-Xcompiler", "-fPIC", *build.ARCH, "-O3", "-std=c++17", "-I", build.CSRC,
                    src, "-o", out, *link, "-lcudart"], check=True)
    return ctypes.CDLL(out)
