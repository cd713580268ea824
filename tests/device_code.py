"""Small CUDA sources of the tests, compiled against the library's headers and loaded with ctypes."""
import ctypes
import os
import subprocess

from paper_2505_24807_gb300 import build, xs

CSRC = build.CSRC


def compile_and_load(tmp, name, source):
    """extern "C" functions of `source` as a shared library linked with libxs."""
    src, out = os.path.join(tmp, name + ".cu"), os.path.join(tmp, name + ".so")
    with open(src, "w") as f:
        f.write(source)
    lib = os.path.dirname(xs.LIB_PATH)
    subprocess.run([build.nvcc(), *build.ARCH, "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-I", CSRC,
                    "-I", os.path.join(os.path.dirname(build.HERE), "include"), "-shared", "-cudart", "shared", src,
                    "-o", out, "-L", lib, "-l:libxs.so", "-Xlinker", "-rpath", "-Xlinker", lib], check=True)
    return ctypes.CDLL(out)
