"""Build ``libspiffy.so`` (nvcc, sm_100a) and its Python binding ``_binding.so``
(the host compiler, against torch's headers) in-tree.

Usage: ``python -m paper_2509_18085_b200.build [--force] [--verbose]``.
"""
from __future__ import annotations

import glob
import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libspiffy.so")
BINDING = os.path.join(HERE, "_binding.so")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3",
    "-std=c++17", "-Xcompiler", "-fPIC", "-shared", "--threads", "0",
    "-I", os.path.join(ROOT, "include"), "-I", CSRC,
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(p) > t for p in deps)


def _build_binding() -> None:
    import sysconfig
    from torch.utils import cpp_extension as ext
    includes = ext.include_paths(device_type="cuda") + [sysconfig.get_paths()["include"], os.path.join(ROOT, "include")]
    tmp = BINDING + f".tmp{os.getpid()}"
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden"]
    for path in includes:
        cmd += ["-isystem", path]
    cmd += ["-o", tmp, os.path.join(CSRC, "binding.cpp"), "-L" + HERE, "-l:libspiffy.so", "-Wl,-rpath,$ORIGIN"]
    for path in ext.library_paths(device_type="cuda"):
        cmd += ["-L" + path]
    cmd += ["-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python"]
    subprocess.run(cmd, check=True)
    os.replace(tmp, BINDING)


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every CUDA source into one shared library and the binding against
    it; returns the library's path."""
    headers = glob.glob(os.path.join(ROOT, "include", "*.h"))
    if force or _stale(LIB, sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + headers):
        nvcc = os.environ.get("NVCC", "nvcc")
        tmp = LIB + f".tmp{os.getpid()}"
        cmd = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-o", tmp] + sources()
        subprocess.run(cmd, check=True)
        os.replace(tmp, LIB)
    if force or _stale(BINDING, [os.path.join(CSRC, "binding.cpp")] + headers):
        _build_binding()
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
