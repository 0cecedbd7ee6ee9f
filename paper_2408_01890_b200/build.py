"""Builds the CUDA library in-tree: `python -m paper_2408_01890_b200.build [--verbose]`.

Two shared objects next to this file: liblisa_b200.so, the library (sm_100a only, no relocatable device code), and
_lisa_binding.so, the native half of binding.py (a CPython extension against torch's headers, no device code).
"""
from __future__ import annotations

import glob
import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
LIB = os.path.join(HERE, "liblisa_b200.so")
EXT = os.path.join(HERE, "_lisa_binding.so")
EXT_KEY = os.path.join(HERE, "_lisa_binding.key")   # what the extension was built against
EXT_SOURCE = os.path.join(HERE, "csrc", "binding_ext.cpp")


def sources():
    return sorted(glob.glob(os.path.join(HERE, "csrc", "*.cu")))


def _stale():
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = sources() + glob.glob(os.path.join(HERE, "csrc", "*.cuh")) + glob.glob(os.path.join(ROOT, "include", "*.h"))
    return any(os.path.getmtime(p) > t for p in deps)


def _binding_key() -> str:
    """What _lisa_binding.so is built against besides its sources: torch's C++ interface and the interpreter's."""
    import torch
    return "torch %s (cxx11 abi %d), python %s\n" % (torch.__version__, int(torch._C._GLIBCXX_USE_CXX11_ABI), sys.version)


def binding_stale() -> bool:
    deps = [EXT_SOURCE] + glob.glob(os.path.join(ROOT, "include", "*.h"))
    if not os.path.exists(EXT) or any(os.path.getmtime(p) > os.path.getmtime(EXT) for p in deps):
        return True
    try:
        with open(EXT_KEY) as f:
            return f.read() != _binding_key()
    except OSError:
        return True


def build_binding(force: bool = False) -> str:
    if not force and not binding_stale():
        return EXT
    import sysconfig

    import torch
    tdir = os.path.dirname(torch.__file__)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    tmp = EXT + ".%d.tmp" % os.getpid()
    subprocess.check_call([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC",
                           "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI),
                           "-I", os.path.join(tdir, "include"), "-I", os.path.join(tdir, "include", "torch", "csrc", "api", "include"),
                           "-I", os.path.join(cuda, "include"), "-I", sysconfig.get_paths()["include"], "-I", os.path.join(ROOT, "include"),
                           EXT_SOURCE, "-o", tmp, "-L", os.path.join(tdir, "lib"),
                           "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda"])
    os.replace(tmp, EXT)
    with open(tmp, "w") as f:
        f.write(_binding_key())
    os.replace(tmp, EXT_KEY)
    return EXT


def build(force: bool = False, verbose: bool = False) -> str:
    build_binding(force)
    if not force and not _stale():
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    tmp = LIB + ".%d.tmp" % os.getpid()
    cmd = [nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17", "--threads", "0",
           "-shared", "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I", os.path.join(HERE, "csrc"),
           "-o", tmp] + sources()
    if verbose:
        cmd.insert(1, "-Xptxas")
        cmd.insert(2, "-v")
    subprocess.check_call(cmd)
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose="--verbose" in sys.argv))
