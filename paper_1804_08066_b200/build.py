"""Build libmqgrad.so (sm_100a) with nvcc and the Python binding (binding_path) with the host compiler, in-tree.

Usage: python paper_1804_08066_b200/build.py [--force] [--verbose]
The shared objects land next to this file; nvcc cross-compiles without a GPU.
"""
import glob
import os
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(os.path.dirname(HERE), "include")
LIB = os.path.join(HERE, "libmqgrad.so")
BINDING_SRC = os.path.join(CSRC, "mqg_binding.cpp")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-shared", "-Xcompiler", "-fPIC", "-I", INCLUDE, "--threads", "4",
]


def binding_path() -> str:
    """The binding's file.  It fits one interpreter and one torch, so both are part of its name: after an upgrade of
    either, the file is not there and is built, instead of a stale one being loaded."""
    import sysconfig

    import torch
    return os.path.join(HERE, "_binding.torch-%s%s" % (torch.__version__, sysconfig.get_config_var("EXT_SUFFIX")))


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale(target, deps):
    return not os.path.exists(target) or any(os.path.getmtime(d) > os.path.getmtime(target) for d in deps)


def _headers():
    return [*glob.glob(os.path.join(INCLUDE, "*.h")), os.path.abspath(__file__)]


def _compile(cmd, target):
    tmp = target + ".tmp.%d" % os.getpid()
    subprocess.run([*cmd, "-o", tmp], check=True)
    os.replace(tmp, target)


def build_binding(force: bool = False) -> str:
    """The native functions of the Python package: torch tensors in, C ABI calls out."""
    binding = binding_path()
    if not force and not _stale(binding, [BINDING_SRC, *_headers()]):
        return binding
    import sysconfig

    import torch
    from torch.utils import cpp_extension
    nvcc = shutil.which(os.environ.get("NVCC", "nvcc")) or "/usr/local/cuda/bin/nvcc"
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(nvcc)))
    include = [sysconfig.get_paths()["include"], os.path.join(cuda, "include"), INCLUDE, *cpp_extension.include_paths()]
    torch_lib = os.path.join(os.path.dirname(torch.__file__), "lib")
    _compile([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden",
              "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI), *("-I" + d for d in include), BINDING_SRC,
              "-L" + HERE, "-l:libmqgrad.so", "-Wl,-rpath,$ORIGIN",
              "-L" + torch_lib, "-ltorch_python", "-ltorch_cpu", "-lc10_cuda", "-lc10"], binding)
    return binding


def build(force: bool = False, verbose: bool = False) -> str:
    deps = [*sources(), *glob.glob(os.path.join(CSRC, "*.cuh")), *glob.glob(os.path.join(CSRC, "*.h")), *_headers()]
    if force or _stale(LIB, deps):
        nvcc = os.environ.get("NVCC", "nvcc")
        _compile([nvcc, *NVCC_FLAGS, *(["-Xptxas", "-v"] if verbose else []), *sources()], LIB)
    build_binding(force)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
