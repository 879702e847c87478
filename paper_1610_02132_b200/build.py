"""Builds libqsgd.so (the C-ABI library with the sm_100a kernels, nvcc) and _qsgd_native.*.so (its Python
binding, g++ against the torch headers) in-tree."""
import glob
import os
import re
import subprocess
import sysconfig

_HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(_HERE, "csrc")
LIB = os.path.join(_HERE, "libqsgd.so")
NATIVE_SRC = os.path.join(CSRC, "python_binding.cpp")

NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-shared", "-Xcompiler", "-fPIC", "--cudart", "shared", "--threads", "0"]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale(target, deps):
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(p) > t for p in deps)


def _headers():
    return glob.glob(os.path.join(_HERE, "..", "include", "*.h"))


def build_library(force=False, verbose=False):
    """Compile every kernel for sm_100a into libqsgd.so; returns the library path."""
    if force or _stale(LIB, sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + _headers()):
        nvcc = os.environ.get("NVCC", "nvcc")
        tmp = LIB + ".tmp%d" % os.getpid()
        cmd = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-o", tmp] + sources()
        subprocess.check_call(cmd)
        os.replace(tmp, LIB)
    return LIB


def native_path():
    """File of the Python binding for the running Python and torch, whose C++ headers it is compiled against: under
    another of either there is no such file, and it is built instead of an old one being loaded."""
    import torch
    key = "torch%s-%d%s" % (torch.__version__, int(torch._C._GLIBCXX_USE_CXX11_ABI), sysconfig.get_config_var("EXT_SUFFIX"))
    return os.path.join(_HERE, "_qsgd_native." + re.sub(r"[^\w.-]", "_", key))


def build_native(force=False):
    """Compile the Python binding; it finds libqsgd.so beside itself and torch's libraries by rpath."""
    native = native_path()
    if force or _stale(native, [NATIVE_SRC] + _headers()):
        import torch
        from torch.utils import cpp_extension
        for old in glob.glob(os.path.join(_HERE, "_qsgd_native.*so")):      # of another torch or Python
            os.remove(old)
        tmp = native + ".tmp%d" % os.getpid()
        inc = cpp_extension.include_paths("cuda") + [sysconfig.get_paths()["include"]]
        libdirs = cpp_extension.library_paths("cuda")
        cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden",
               "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI)]
        cmd += ["-isystem" + p for p in inc] + [NATIVE_SRC, "-o", tmp]
        cmd += ["-L" + _HERE, "-l:libqsgd.so", "-Wl,-rpath,$ORIGIN"]
        cmd += ["-L" + p for p in libdirs] + ["-Wl,-rpath," + libdirs[0]]
        cmd += ["-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda"]
        subprocess.check_call(cmd)
        os.replace(tmp, native)
    return native


def build(force=False, verbose=False):
    """Builds whatever is out of date; returns the path of libqsgd.so."""
    build_library(force, verbose)
    build_native(force)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose=True))
