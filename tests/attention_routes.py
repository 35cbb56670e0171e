"""Which kernels a tensor-core attention call takes, without a GPU: the library's own launcher, compiled
against a runtime that writes down what is launched (tests/host_runtime/runtime.cpp, 148 multiprocessors)."""
import ctypes
import functools
import os
import re
import shutil
import subprocess
import tempfile

from paper_2509_18085_b200 import build as builder
from paper_2509_18085_b200 import spiffy

HERE = os.path.dirname(os.path.abspath(__file__))
UNITS = ["attention_tc", "attention_pair", "api", "decide", "walk", "stage", "step_host"]


@functools.lru_cache(maxsize=None)
def _library():
    out = tempfile.mkdtemp(prefix="attention_routes")
    inc = ["-I", os.path.join(builder.ROOT, "include"), "-I", builder.CSRC]
    cuda = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    obj = {u: os.path.join(out, u + ".o") for u in UNITS}
    jobs = [subprocess.Popen([os.environ.get("NVCC", "nvcc"), "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17",
                              "-Xcompiler", "-fPIC", "-c", os.path.join(builder.CSRC, u + ".cu"), "-o", obj[u]] + inc)
            for u in UNITS]
    assert [j.wait() for j in jobs] == [0] * len(jobs)
    so = os.path.join(out, "routes.so")
    subprocess.run([os.environ.get("CXX", "g++"), "-std=c++17", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-DREAL_ATTENTION",
                    "-isystem", cuda] + inc + [os.path.join(HERE, "host_runtime", "runtime.cpp")] + list(obj.values()) +
                   ["-o", so], check=True)
    lib = ctypes.CDLL(so)
    shutil.rmtree(out)
    lib.fake_log.restype = ctypes.c_char_p
    lib.fake_reset.argtypes = [ctypes.c_char_p, ctypes.c_size_t, ctypes.c_size_t]
    return lib


def _launches(lib):
    out = []
    for line in lib.fake_log().decode().splitlines():
        blocks, cluster = (int(n) for n in re.search(r"blocks (\d+) cluster (\d+)$", line).groups())
        if "graph_attention_pair_kernel" in line:
            name = "pair"
        else:
            nq = int(re.search(r"graph_attention_tc_kernelILi(\d)", line).group(1))
            name = "two tiles" if nq == 2 else "one tile" if cluster == 1 else f"cluster of {cluster}"
        out.append((name, blocks))
    return out


def launches(B, N, L, P, Hq, Hkv, d=128, flags=0):
    """[(route, thread blocks)] of a call's launches: "pair" (of thread blocks to an M-tile), "one tile" or "two
    tiles" (M-tiles per thread block), "cluster of 2" (4, 8: thread blocks that share an M-tile's key tiles)."""
    lib, p = _library(), ctypes.c_void_p(1 << 20)
    lib.fake_reset(b"", 0, 0)
    desc = spiffy.AttnDesc(B, N, L, P, Hq, Hkv, d, spiffy.BF16, 0.0, spiffy.ATTN_AUTO | flags)
    assert lib.spiffy_graph_attention(ctypes.byref(desc), *[p] * 7, None, ctypes.c_size_t(0), None) == spiffy.OK
    return _launches(lib)


def route(*shape, **more):
    return ", then ".join(name for name, _ in launches(*shape, **more))


def full_sequence_route(B, N, L, P, S, Hq, Hkv):
    lib, p = _library(), ctypes.c_void_p(1 << 20)
    lib.fake_reset(b"", 0, 0)
    desc = spiffy.AttnDesc(B, N, L, P, Hq, Hkv, 128, spiffy.BF16, 0.0, spiffy.ATTN_AUTO)
    assert lib.spiffy_full_sequence_attention(ctypes.byref(desc), S, *[p] * 11, None, ctypes.c_size_t(0), None) == spiffy.OK
    return ", then ".join(name for name, _ in _launches(lib))
