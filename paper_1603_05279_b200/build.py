"""Builds libxnor.so (the C-ABI CUDA library) in-tree with nvcc for sm_100a, and beside it
_pymarshal.so, the native half of the Python binding."""
import glob
import os
import subprocess
import sysconfig

_HERE = os.path.dirname(os.path.abspath(__file__))
_ROOT = os.path.dirname(_HERE)
LIB = os.path.join(_HERE, "libxnor.so")
LIB_CHECK = os.path.join(_HERE, "libxnor_check.so")     # the same sources with -DXNOR_BOUNDS_CHECK
SOURCES = sorted(glob.glob(os.path.join(_HERE, "csrc", "*.cu")))
HEADERS = sorted(glob.glob(os.path.join(_HERE, "csrc", "*.cuh"))) + \
    sorted(glob.glob(os.path.join(_ROOT, "include", "*.h")))

PYEXT = os.path.join(_HERE, "_pymarshal.so")
PYEXT_SOURCE = os.path.join(_HERE, "csrc", "pymarshal.cpp")

NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-t", "8", "-Xcompiler", "-fPIC", "-shared", "-I", os.path.join(_ROOT, "include")]


def up_to_date(lib=LIB):
    if not os.path.exists(lib):
        return False
    t = os.path.getmtime(lib)
    return all(os.path.getmtime(f) <= t for f in SOURCES + HEADERS)


def build_pyext(force=False):
    """Builds _pymarshal.so against the installed torch (its libraries are loaded by then)."""
    inputs = [PYEXT_SOURCE] + glob.glob(os.path.join(_ROOT, "include", "*.h"))
    if not force and os.path.exists(PYEXT) and \
            all(os.path.getmtime(f) <= os.path.getmtime(PYEXT) for f in inputs):
        return PYEXT
    import torch
    troot = os.path.dirname(torch.__file__)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared",
           "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI),
           "-I", os.path.join(_ROOT, "include"), "-I", sysconfig.get_paths()["include"]]
    for inc in (os.path.join(troot, "include"), os.path.join(troot, "include/torch/csrc/api/include"),
                os.path.join(cuda, "include")):
        cmd += ["-isystem", inc]
    cmd += [PYEXT_SOURCE, "-o", PYEXT, "-L", os.path.join(troot, "lib"),
            "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda"]
    subprocess.run(cmd, check=True)
    return PYEXT


def build_library(force=False, verbose=False, bounds_check=False):
    """Builds libxnor.so, or with bounds_check the checking build libxnor_check.so: nvcc alone."""
    lib = LIB_CHECK if bounds_check else LIB
    if not force and up_to_date(lib):
        return lib
    nvcc = os.environ.get("NVCC", "nvcc")
    cmd = [nvcc] + NVCC_FLAGS + (["-DXNOR_BOUNDS_CHECK"] if bounds_check else []) + \
        (["-Xptxas", "-v"] if verbose else []) + ["-o", lib] + SOURCES
    subprocess.run(cmd, check=True)
    return lib


def build(force=False, verbose=False, bounds_check=False):
    """The library, and then the Python binding's native half: the C library needs neither torch's headers
    nor a host C++ compiler set up for them, and is there when building the other fails."""
    lib = build_library(force, verbose, bounds_check)
    build_pyext(force and not bounds_check)
    return lib


if __name__ == "__main__":
    print(build(force=True, verbose=True))
