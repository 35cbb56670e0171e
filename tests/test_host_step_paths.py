"""The host code of the host-buffer step and of the decision without a GPU: compiled
against a runtime that logs what it is asked for (tests/host_runtime/runtime.cpp) and
fails where told."""
import ctypes
import os
import re
import subprocess

import pytest
import torch

from paper_2509_18085_b200 import build as builder
from paper_2509_18085_b200 import spiffy
from paper_2509_18085_b200 import workloads as W
from paper_2509_18085_b200.step import VerifyStep, inputs_from_workload

HERE = os.path.dirname(os.path.abspath(__file__))
UNITS = ["step_host", "decide", "walk", "draft", "stage", "api"]


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    """The library's host code with the stand-in runtime."""
    out = tmp_path_factory.mktemp("host")
    inc = ["-I", os.path.join(builder.ROOT, "include"), "-I", builder.CSRC]
    cuda = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    jobs = [subprocess.Popen([os.environ.get("NVCC", "nvcc"), "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17",
                              "-Xcompiler", "-fPIC", "-c", os.path.join(builder.CSRC, u + ".cu"), "-o",
                              str(out / (u + ".o"))] + inc) for u in UNITS]
    assert [j.wait() for j in jobs] == [0] * len(jobs)
    so = out / "host.so"
    subprocess.run([os.environ.get("CXX", "g++"), "-std=c++17", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-isystem", cuda] + inc +
                   [os.path.join(HERE, "host_runtime", "runtime.cpp")] + [str(out / (u + ".o")) for u in UNITS] +
                   ["-o", str(so)], check=True)
    lib = ctypes.CDLL(str(so))
    lib.fake_log.restype = ctypes.c_char_p
    lib.fake_reset.argtypes = [ctypes.c_char_p, ctypes.c_size_t, ctypes.c_size_t]
    lib.spiffy_verify_step_host_workspace.restype = ctypes.c_size_t
    return lib


STREAM = 7
BASE, STEP = 1 << 32, 1 << 24  # the host arrays: never touched, only told apart
NAMES = ["q", "k_prefix", "v_prefix", "k_block", "v_block", "logits", "block_tokens", "parent_off", "parent_idx",
         "accepted_node", "n_accepted", "path", "next_block", "status"]


def desc(N=4, L=8, d=128, dtype=spiffy.BF16, kernel=spiffy.ATTN_AUTO, cap=4, V=1024, Hq=4, Hkv=4):
    return spiffy.StepDesc(spiffy.AttnDesc(1, N, L, 16, Hq, Hkv, d, dtype, 0.0, kernel),
                           spiffy.DecideDesc(1, N, L, V, dtype, V, V - 1, spiffy.RULE_TOPS, 1, 0.9), cap)


def step(lib, d, fail="", pinned=True, **moved):
    """(status, log lines) of one call."""
    lib.fake_reset(fail.encode(), BASE if pinned else 0, BASE + 100 * STEP if pinned else 0)
    at = {n: BASE + i * STEP for i, n in enumerate(NAMES)}
    at.update({n: at[n] + by for n, by in moved.items()})
    st = lib.spiffy_verify_step_host(ctypes.byref(d), *(ctypes.c_void_p(at[n]) for n in NAMES),
                                     ctypes.c_void_p(1 << 20), ctypes.c_size_t(1 << 40), ctypes.c_void_p(STREAM))
    return st, lib.fake_log().decode().splitlines()


def busy_streams(log):
    """Streams that hold work nobody has waited for when the call returns."""
    busy = set()
    for line in log:
        s = int(re.search(r" on (\d+)", line).group(1))
        if line.startswith("sync"):
            busy.discard(s)
        elif line.startswith(("memcpy", "memset", "launch")) and not line.endswith("FAILED"):
            busy.add(s)
    return busy


@pytest.mark.parametrize("bad", [dict(d=96), dict(kernel=spiffy.ATTN_TCGEN05, d=64),
                                 dict(kernel=spiffy.ATTN_TCGEN05, dtype=spiffy.F32), dict(Hkv=3), dict(kernel=9)])
@pytest.mark.parametrize("pinned", [True, False])
def test_a_refused_step_enqueues_nothing(host, bad, pinned):
    st, log = step(host, desc(**bad), pinned=pinned)
    assert st in (spiffy.EINVAL, spiffy.EUNSUPPORTED)
    assert log == []


@pytest.mark.parametrize("pinned", [True, False])
@pytest.mark.parametrize("dtype", [spiffy.BF16, spiffy.F32])
def test_nothing_is_in_flight_when_a_step_fails(host, dtype, pinned):
    """Whatever call fails, the caller's arrays and workspace are at rest when it hears of it."""
    st, log = step(host, desc(dtype=dtype), pinned=pinned)
    assert st == spiffy.OK
    kinds = {re.sub(r"( on \d+).*", r"\1", line) for line in log if not line.startswith("sync")}
    assert any(k.startswith("launch attention") for k in kinds)
    for kind in sorted(kinds):
        st, log = step(host, desc(dtype=dtype), fail=kind, pinned=pinned)
        assert st == spiffy.ECUDA, kind
        assert busy_streams(log) == set(), (kind, log)


@pytest.mark.parametrize("by", [2, 8])
def test_kernels_read_pinned_logits_only_on_16_byte_boundaries(host, by):
    """Elsewhere their vector loads would be misaligned: the runtime copies all rows."""
    d = desc()
    for pinned_lists in (True, False):  # would be read in place; would be staged by a kernel
        moved = dict(logits=by) if pinned_lists else dict(logits=by, parent_off=100 * STEP)
        st, log = step(host, d, **moved)
        assert st == spiffy.OK
        assert not any("stage_masked_rows" in line for line in log)
        src = BASE + NAMES.index("logits") * STEP + by
        assert any(line.startswith("memcpy") and f"from {src} bytes {4 * 8 * 1024 * 2}" in line for line in log)


@pytest.mark.parametrize("flags", [0x100, 0x200, 0x400, 0x700])
@pytest.mark.parametrize("pinned", [True, False])
def test_flags_of_the_component_calls_change_nothing(host, flags, pinned):
    """Least of all the size of a logits element, which sizes the staging and its copies."""
    want = step(host, desc(), pinned=pinned)
    flagged = desc()
    flagged.decide.logits_dtype |= flags
    flagged.attn.kernel |= flags & 0x300
    assert host.spiffy_verify_step_host_workspace(ctypes.byref(flagged)) == \
        host.spiffy_verify_step_host_workspace(ctypes.byref(desc()))
    assert step(host, flagged, pinned=pinned) == want


@pytest.mark.parametrize("N,L", [(200, 20), (16, 32)])  # separate walk; fused tail
def test_lists_are_left_in_host_memory_only_where_they_are_read_once(host, N, L):
    """Around the largest graph that the walk copies to shared memory: 40 KB."""
    edge = 40 * 1024 // 4 - (2 * N * L + 4 * N + 1)
    lists = str(BASE + NAMES.index("parent_off") * STEP)
    for cap in (edge - 1, edge, edge + 1, edge + N, edge + N + 1):
        st, log = step(host, desc(N=N, L=L, cap=cap))
        assert st == spiffy.OK
        (walk,) = [line for line in log if "accept_walk" in line or "decide_tail" in line]
        in_place = f" lists {lists} " in walk
        assert in_place == (cap <= edge), (cap - edge, walk)
        assert not in_place or "decide_tail" in walk or walk.endswith("staged 1")


@pytest.mark.parametrize("N,L,cap", [(4, 8, 4), (16, 32, 4), (54, 32, 4), (3, 8, 14000)])
def test_an_independent_kernel_may_start_as_the_reduce_ends(host, N, L, cap):
    """SPIFFY_INDEPENDENT_NEXT on both routes: every kernel of the call lets its dependents start ahead
    of its own wait, so that what follows moves in behind the reduce.  (The fused tail does anyway
    once it has waited, the small kernels of the other route at once.)"""
    fused = N * L <= 512 and cap < 10000
    d = spiffy.DecideDesc(1, N, L, 1024, spiffy.BF16, 1024, 1023, spiffy.RULE_TOPS, 1, 0.9)
    p = ctypes.c_void_p(1 << 20)
    for flags, early in ((0, "0"), (spiffy.INDEPENDENT_NEXT, "1")):
        d.logits_dtype = spiffy.BF16 | flags
        host.fake_reset(b"", 0, 0)
        assert host.spiffy_decide_walk(ctypes.byref(d), p, p, p, p, cap, *[p] * 11, ctypes.c_size_t(1 << 40),
                                       ctypes.c_void_p(STREAM)) == spiffy.OK
        log = host.fake_log().decode().splitlines()
        assert len(log) == (2 if fused else 3)
        assert log[0].endswith(f" early {'1' if fused else early}")
        if fused:  # the tail is resident while the reduce runs either way
            assert log[1].endswith(f" early {early}")


@pytest.mark.parametrize("flags", [0, spiffy.INDEPENDENT, spiffy.INDEPENDENT_NEXT])
@pytest.mark.parametrize("N,L,V,dtype", [
    (16, 32, 8 * 8192, spiffy.BF16), (16, 32, 8 * 8192 + 8, spiffy.BF16),        # 512 rows of 8 slices, of 9
    (8, 32, 16 * 8192, spiffy.BF16), (8, 32, 16 * 8192 + 8, spiffy.BF16),
    (3, 13, 105 * 4096, spiffy.F32), (3, 13, 105 * 4096 + 4, spiffy.F32),        # 39 rows of 105, of 106
    (9, 57, 1000, spiffy.BF16), (16, 32, 1000, spiffy.BF16)])                    # 513 rows, and 512, of one
def test_fused_tail_up_to_4096_partial_results(host, N, L, V, dtype, flags):
    """Beyond, the kernels apart, unless an attention comes next and the merging runs beside it."""
    slices = -(-V // (8192 if dtype == spiffy.BF16 else 4096))
    fused = N * L <= 512 and (N * L * slices <= 4096 or flags == spiffy.INDEPENDENT_NEXT)
    d = spiffy.DecideDesc(1, N, L, V, dtype | flags, V, V - 1, spiffy.RULE_TOPS, 1, 0.9)
    p = ctypes.c_void_p(1 << 20)
    host.fake_reset(b"", 0, 0)
    assert host.spiffy_decide_walk(ctypes.byref(d), p, p, p, p, 4, *[p] * 11, ctypes.c_size_t(1 << 40),
                                   ctypes.c_void_p(STREAM)) == spiffy.OK
    kernels = [re.search("(decide_reduce|decide_tail|decide_finalize|accept_walk)_kernel", line).group(1) for line in host.fake_log().decode().splitlines()]
    assert kernels == (["decide_reduce", "decide_tail"] if fused else ["decide_reduce", "decide_finalize", "accept_walk"])


@pytest.mark.parametrize("B,N,L,fit", [(1, 4, 8, 1), (148, 8, 8, 1), (149, 16, 27, 2), (149, 8, 16, 4), (600, 8, 8, 4), (65535, 1, 1, 4)])
def test_tails_of_more_sequences_than_multiprocessors_share_them(host, B, N, L, fit):
    """65536 registers at 48 a thread, 148 multiprocessors."""
    d = spiffy.DecideDesc(B, N, L, 1024, spiffy.BF16, 1024, 1023, spiffy.RULE_TOPS, 1, 0.9)
    p = ctypes.c_void_p(1 << 20)
    host.fake_reset(b"", 0, 0)
    assert host.spiffy_decide_walk(ctypes.byref(d), p, p, p, p, 4, *[p] * 11, ctypes.c_size_t(1 << 40),
                                   ctypes.c_void_p(STREAM)) == spiffy.OK
    (tail,) = [line for line in host.fake_log().decode().splitlines() if "decide_tail" in line]
    assert 65536 // (48 * int(re.search(r"threads (\d+)", tail).group(1))) >= fit


@pytest.mark.parametrize("B,N,L,threads", [(9, 4, 8, 256), (32, 8, 8, 256), (20, 9, 2, 512), (9, 5, 13, 512), (9, 16, 8, 512),
                                           (9, 17, 1, 1024), (9, 3, 43, 1024), (120, 16, 32, 1024)])
@pytest.mark.parametrize("flags", [0, spiffy.INDEPENDENT, spiffy.INDEPENDENT_NEXT])
def test_a_tail_is_no_larger_than_its_graph_asks_for(host, B, N, L, threads, flags):
    """A warp per node, four threads a row: the attention beside it leaves no room for more."""
    d = spiffy.DecideDesc(B, N, L, 1024, spiffy.F32 | flags, 1024, 1023, spiffy.RULE_TOPS, 1, 0.9)
    p = ctypes.c_void_p(1 << 20)
    host.fake_reset(b"", 0, 0)
    assert host.spiffy_decide_walk(ctypes.byref(d), p, p, p, p, 4, *[p] * 11, ctypes.c_size_t(1 << 40),
                                   ctypes.c_void_p(STREAM)) == spiffy.OK
    (tail,) = [line for line in host.fake_log().decode().splitlines() if "decide_tail" in line]
    assert int(re.search(r"threads (\d+)", tail).group(1)) == threads


@pytest.mark.parametrize("B,N,L,V,dtype,cap,small", [
    (1, 1, 1, 100, spiffy.F32, 4, True), (8, 4, 16, 4096, spiffy.F32, 4, True), (9, 4, 16, 4096, spiffy.F32, 4, False),
    (1, 8, 8, 8192, spiffy.BF16, 4, True), (1, 8, 8, 8200, spiffy.BF16, 4, False), (2, 13, 5, 1000, spiffy.BF16, 4, False),
    (1, 2, 8, 16384, spiffy.F32, 4, True), (1, 2, 8, 16388, spiffy.F32, 4, False), (1, 4, 8, 1024, spiffy.F32, 11000, True),
    (1, 4, 8, 1024, spiffy.F32, 12000, False)])
@pytest.mark.parametrize("flags", [0, spiffy.INDEPENDENT, spiffy.INDEPENDENT_NEXT, spiffy.INDEPENDENT | spiffy.INDEPENDENT_NEXT])
def test_up_to_64_slices_beside_an_attention_are_one_launch(host, B, N, L, V, dtype, cap, small, flags):
    d = spiffy.DecideDesc(B, N, L, V, dtype | flags, V, V - 1, spiffy.RULE_TOPS, 1, 0.9)
    p = ctypes.c_void_p(1 << 20)
    host.fake_reset(b"", 0, 0)
    assert host.spiffy_decide_walk(ctypes.byref(d), p, p, p, p, cap, *[p] * 11, ctypes.c_size_t(1 << 40),
                                   ctypes.c_void_p(STREAM)) == spiffy.OK
    log = host.fake_log().decode().splitlines()
    assert (["decide_small" in line for line in log] == [True]) == (small and bool(flags & spiffy.INDEPENDENT))


@pytest.mark.parametrize("D,L", [(1, 1), (64, 1), (1000, 1), (300, 4), (10, 15), (1000, 17), (10, 32), (10, 33), (1024, 64)])
def test_drafting_has_threads_for_positions_and_formulas(host, D, L):
    """A warp per position, two positions a warp beyond 32; on short blocks 512 threads for the formulas all the same."""
    d = spiffy.DraftDesc(1, L, 1000, spiffy.F32, 1000, 999, D, 1, 1, 8)
    p = ctypes.c_void_p(1 << 20)
    host.fake_reset(b"", 0, 0)
    assert host.spiffy_draft_blocks(ctypes.byref(d), *[p] * 14, ctypes.c_size_t(1 << 40), ctypes.c_void_p(STREAM)) == spiffy.OK
    (build,) = [line for line in host.fake_log().decode().splitlines() if "draft_build" in line]
    threads = int(re.search(r"threads (\d+)", build).group(1))
    assert 512 <= threads <= 1024 and threads % 32 == 0 and threads >= 32 * min(L, 32)


@pytest.mark.parametrize("B,D,L,threads", [(1, 64, 8, 512), (1, 65, 1, 1024), (148, 1000, 16, 1024), (149, 1000, 16, 512),
                                           (149, 1000, 17, 544)])
def test_drafting_of_large_graphs_has_all_threads(host, B, D, L, threads):
    """While there is a multiprocessor for every sequence."""
    d = spiffy.DraftDesc(B, L, 1000, spiffy.F32, 1000, 999, D, 1, 1, 8)
    p = ctypes.c_void_p(1 << 20)
    host.fake_reset(b"", 0, 0)
    assert host.spiffy_draft_blocks(ctypes.byref(d), *[p] * 14, ctypes.c_size_t(1 << 40), ctypes.c_void_p(STREAM)) == spiffy.OK
    (build,) = [line for line in host.fake_log().decode().splitlines() if "draft_build" in line]
    assert int(re.search(r"threads (\d+)", build).group(1)) == threads


def test_a_step_object_describes_each_input_anew(monkeypatch):
    """The parent lists of one graph are longer than the next one's: a descriptor kept from the first
    call would read past the end of the second call's arrays."""
    seen = []
    monkeypatch.setattr(torch.Tensor, "pin_memory", lambda t: t)
    monkeypatch.setattr(spiffy, "spiffy_verify_step_host", lambda d, *a: seen.append((d.parent_cap, a[-1].numel())))
    cfg = W.Config("t", 2, 4, 8, 16, 4, 4, 64, "bf16", 1000, spiffy.RULE_TOPS)
    step, x = VerifyStep(cfg, device="cpu"), inputs_from_workload(W.make(cfg, 3), device="cpu")
    for cap in (40, 4, 4000):
        x.parent_idx = torch.zeros((2, cap), dtype=torch.int32)
        step.run_host(x)
    assert [cap for cap, _ in seen] == [40, 4, 4000]
    assert seen[0][1] == seen[1][1] < seen[2][1]  # the workspace grows, and is otherwise kept


def test_poll_limits_leave_time_for_products_in_flight(host):
    """None at all, or at least 16384 polls: far more than a group of tensor-core products takes."""
    limit = getattr(host, "_ZN6spiffy15mbar_poll_limitEv")
    limit.restype = ctypes.c_uint32
    set_limits = host.spiffy_set_wait_limits
    set_limits.argtypes = [ctypes.c_int64, ctypes.c_int64, ctypes.c_int32]
    for asked, got in ((0, 0), (1, 1 << 14), (3000, 1 << 14), (1 << 14, 1 << 14), (100000, 100000), (1 << 40, 1 << 20), (-1, 1 << 20)):
        set_limits(asked, -1, 0)
        assert limit() == got
