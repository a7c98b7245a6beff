"""Compiles small C++ helpers against the library's internal headers, for tests of
host-side choices that the C ABI does not show."""
import ctypes
import os
import subprocess

from paper_1406_1864_gb300 import build as B


def compile_helper(source: str, folder) -> ctypes.CDLL:
    lib = B.build()
    src, so = os.path.join(str(folder), "helper.cpp"), os.path.join(str(folder), "helper.so")
    with open(src, "w") as f:
        f.write(source)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.check_call(["g++", "-std=c++17", "-shared", "-fPIC", f"-I{cuda}/include", "-I",
                           os.path.join(B.ROOT, "include"), "-I", B.CSRC, src, "-L", B.HERE,
                           "-l:" + os.path.basename(lib), f"-Wl,-rpath,{B.HERE}", "-o", so])
    return ctypes.CDLL(so)
