"""Build the C-ABI library ``libspqt.so`` in-tree with nvcc for sm_100a, and ``_native.<Python>.<PyTorch>.so``, the Python
marshalling of its per-token calls (``csrc/spqt_python.cpp``), with g++ against PyTorch's headers.

    python -m paper_2511_04477_b200.build [--force] [--verbose]

nvcc cross-compiles without a GPU.  The shared objects are written next to this
file so that they travel with the source tree.
"""
from __future__ import annotations

import glob
import os
import subprocess
import sys

_HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(_HERE, "csrc")
LIB_PATH = os.path.join(_HERE, "libspqt.so")
NATIVE_SOURCE = os.path.join(CSRC, "spqt_python.cpp")
HEADER = os.path.join(os.path.dirname(_HERE), "include", "spqt.h")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a",
    "-O3", "-lineinfo", "-std=c++17", "--threads", "0",
    "-Xcompiler", "-fPIC", "-shared",
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def _run(cmd, tmp: str, target: str, verbose: bool) -> None:
    res = subprocess.run(cmd, capture_output=True, text=True)
    if verbose:
        sys.stderr.write(res.stderr)
    if res.returncode != 0:
        raise RuntimeError("%s failed:\n%s\n%s" % (cmd[0], " ".join(cmd), res.stderr))
    os.replace(tmp, target)


def _build_native(target: str, verbose: bool) -> None:
    import sysconfig

    import torch
    from torch.utils import cpp_extension

    root = os.path.dirname(torch.__file__)
    cuda = cpp_extension.CUDA_HOME or "/usr/local/cuda"
    includes = [os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"),
                os.path.join(cuda, "include"), sysconfig.get_paths()["include"]]
    tmp = target + ".%d.tmp" % os.getpid()
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
           "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI)]
    for d in includes:
        cmd += ["-isystem", d]
    cmd += [NATIVE_SOURCE, "-o", tmp, "-L" + _HERE, "-l:libspqt.so", "-Wl,-rpath,$ORIGIN",
            "-L" + os.path.join(root, "lib"), "-ltorch_python", "-ltorch_cuda", "-ltorch_cpu", "-lc10_cuda", "-lc10"]
    _run(cmd, tmp, target, verbose)


def build(force: bool = False, verbose: bool = False) -> str:
    if force or _stale(LIB_PATH, sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + [HEADER]):
        tmp = LIB_PATH + ".%d.tmp" % os.getpid()
        _run([os.environ.get("NVCC", "nvcc")] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-o", tmp] + sources(),
             tmp, LIB_PATH, verbose)
    from .binding import native_path

    native = native_path()
    if force or _stale(native, [NATIVE_SOURCE, HEADER]):
        _build_native(native, verbose)
    return LIB_PATH


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
