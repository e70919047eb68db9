"""Build libmate.so (nvcc, sm_100a; cross-compiles without a GPU) and the native Python binding in-tree."""
import glob
import os
import shutil
import subprocess
import sys
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
LIB = os.path.join(PKG, "libmate.so")
BINDING = os.path.join(CSRC, "binding.cpp")
NATIVE = os.path.join(PKG, "_native.so")
TRACE_LIB = os.path.join(PKG, "libmate_trace.so")   # same sources with -DMATE_TRACE (cycle counters per role)


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _deps():
    return sources() + glob.glob(os.path.join(CSRC, "*.h")) + glob.glob(os.path.join(CSRC, "*.cuh")) + \
        [os.path.join(ROOT, "include", "mate.h")]


def build_binding(force: bool = False) -> str:
    """The native module of the Python binding (host code against torch's C++ headers; libmate is not linked)."""
    deps = [BINDING, os.path.join(ROOT, "include", "mate.h")]
    if not force and os.path.exists(NATIVE) and all(os.path.getmtime(p) <= os.path.getmtime(NATIVE) for p in deps):
        return NATIVE
    import torch
    from torch.utils import cpp_extension
    tmp = NATIVE + ".%d.tmp" % os.getpid()
    cuda = os.environ.get("CUDA_HOME") or os.path.dirname(os.path.dirname(os.path.realpath(shutil.which("nvcc") or
                                                                                           "/usr/local/cuda/bin/nvcc")))
    include = [os.path.join(ROOT, "include"), sysconfig.get_paths()["include"], os.path.join(cuda, "include")] + \
        cpp_extension.include_paths()
    libs = os.path.join(os.path.dirname(torch.__file__), "lib")
    subprocess.run([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden",
                    "-D_GLIBCXX_USE_CXX11_ABI=%d" % torch._C._GLIBCXX_USE_CXX11_ABI]
                   + ["-I" + d for d in include] + ["-o", tmp, BINDING, "-L" + libs, "-Wl,-rpath," + libs]
                   + ["-l" + x for x in ("c10", "c10_cuda", "torch_cpu", "torch_cuda", "torch_python")], check=True)
    os.replace(tmp, NATIVE)
    return NATIVE


def build(force: bool = False, verbose: bool = False, trace: bool = False) -> str:
    """Compiles the library (trace=True: the profiling build with cycle counters, libmate_trace.so,
    which `bench.py --trace` loads; it is a few per cent slower and never the default)."""
    build_binding(force)
    lib = TRACE_LIB if trace else LIB
    if not force and os.path.exists(lib):
        t = os.path.getmtime(lib)
        if all(os.path.getmtime(p) <= t for p in _deps()):
            return lib
    nvcc = os.environ.get("NVCC", "nvcc")
    tmp = lib + ".%d.tmp" % os.getpid()
    cmd = [nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
           "-shared", "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I", CSRC,
           "-o", tmp] + sources()
    if trace:
        cmd.insert(1, "-DMATE_TRACE")
    if verbose:
        cmd.insert(1, "-Xptxas")
        cmd.insert(2, "-v")
    subprocess.run(cmd, check=True)
    os.replace(tmp, lib)
    return lib


if __name__ == "__main__":
    print(build(force=True, verbose="-v" in sys.argv, trace="--trace" in sys.argv))
