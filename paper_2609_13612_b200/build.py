"""Build libattnfuse.so (sm_100a, nvcc) and the torch binding (g++) in-tree.  `python -m paper_2609_13612_b200.build`."""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(PKG, "csrc")
LIB = os.path.join(PKG, "libattnfuse.so")
BINDING = os.path.join(PKG, "_torch_binding.so")
BINDING_SRC = os.path.join(CSRC, "torch_binding.cpp")
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-shared", "-Xcompiler", "-fPIC"]


def _sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")) +
                  [os.path.join(os.path.dirname(PKG), "include", "attnfuse.h")])


def is_stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    return any(os.path.getmtime(s) > t for s in _sources())


def abi_tag() -> str:
    """What the native binding depends on: it is built for one Python and one torch."""
    import torch
    return "built for Python %d.%d, torch %s" % (sys.version_info[0], sys.version_info[1], torch.__version__)


def binding_is_stale() -> bool:
    deps = [BINDING_SRC, os.path.join(os.path.dirname(PKG), "include", "attnfuse.h")]
    if not os.path.exists(BINDING) or any(os.path.getmtime(d) > os.path.getmtime(BINDING) for d in deps):
        return True
    with open(BINDING, "rb") as f:
        return abi_tag().encode() + b"\0" not in f.read()


def build_binding(force: bool = False) -> str:
    """The native side of the Python binding: a CPython module over torch's C++ headers, host code only."""
    if not force and not binding_is_stale():
        return BINDING
    import torch
    root = os.path.dirname(os.path.abspath(torch.__file__))
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    inc = [os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"),
           sysconfig.get_paths()["include"], os.path.join(cuda, "include")]
    tmp = BINDING + ".tmp.%d" % os.getpid()
    subprocess.check_call([os.environ.get("CXX", "g++"), "-O2", "-std=c++20", "-shared", "-fPIC", "-fvisibility=hidden",
                           "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI), '-DAF_ABI_TAG="%s"' % abi_tag()] +
                          ["-isystem" + d for d in inc] + ["-o", tmp, BINDING_SRC, "-L" + os.path.join(root, "lib"),
                           "-Wl,-rpath," + os.path.join(root, "lib"), "-ltorch_python", "-ltorch_cuda", "-ltorch_cpu", "-lc10_cuda", "-lc10"])
    os.replace(tmp, BINDING)
    return BINDING


def build(force: bool = False, verbose: bool = False) -> str:
    build_binding(force)
    if not force and not is_stale():
        return LIB
    nvcc = os.environ.get("NVCC", "nvcc")
    tmp = LIB + ".tmp.%d" % os.getpid()
    cmd = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + \
          ["-o", tmp, os.path.join(CSRC, "attnfuse.cu")]
    subprocess.check_call(cmd)
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    import sys
    print(build(force=True, verbose="-v" in sys.argv))
