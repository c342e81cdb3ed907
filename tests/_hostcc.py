"""Compile functions of the library's __host__ __device__ headers for the host."""
import ctypes
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1808_06194_gb300", "csrc")


def host_lib(folder, name, code):
    """The shared library of C++ source `code`, which may include headers of csrc/."""
    src, so = os.path.join(str(folder), name + ".cpp"), os.path.join(str(folder), name + ".so")
    with open(src, "w") as f:
        f.write(code)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-D__host__=", "-D__device__=",
                    "-D__constant__=", "-I", CSRC, "-I", os.path.join(ROOT, "include"), src, "-o", so], check=True)
    return ctypes.CDLL(so)
