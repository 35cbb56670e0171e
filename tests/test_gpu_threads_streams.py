"""The calls among other threads and streams of the caller's program."""
import threading
import time

import pytest
import torch

from paper_2509_18085_b200 import spiffy
from paper_2509_18085_b200 import workloads as W
import gpu_util as G

pytestmark = pytest.mark.gpu


def small(B=1, N=3, L=5, V=1000):
    cfg = W.Config("t", dtype="f32", vocab=V, rule=spiffy.RULE_TOPS, batch=B, n_nodes=N, block_len=L, prefix_len=0,
                   n_q_heads=1, n_kv_heads=1, head_dim=64)
    w = W.make(cfg, 5, attention=False)
    return cfg, [G.to_dev(a) for a in (w.logits, w.block_tokens, w.parent_off, w.parent_idx)]


def test_a_full_launch_queue_stops_only_the_thread_that_launches():
    """About a thousand launches fit a stream's queue; whoever adds more waits for the device, here for
    half a second, and the other threads of the process go on."""
    cfg, (lg, tk, off, idx) = small()
    spiffy.spiffy_decide_walk(lg, tk, off, idx, cfg.mask_id, cfg.rule)
    torch.cuda.synchronize()
    spent = []

    def fill():
        torch.cuda._sleep(1_000_000_000)
        t = time.perf_counter()
        for _ in range(1200):  # two or three launches each
            spiffy.spiffy_decide_walk(lg, tk, off, idx, cfg.mask_id, cfg.rule)
        spent.append(time.perf_counter() - t)

    thread = threading.Thread(target=fill)
    longest, last = 0.0, time.perf_counter()
    thread.start()
    while thread.is_alive():
        time.sleep(1e-3)
        now = time.perf_counter()
        longest, last = max(longest, now - last), now
    thread.join()
    torch.cuda.synchronize()
    assert spent[0] > 0.25, "the queue never filled up: this shows nothing"
    assert longest < 0.1, f"another thread stood still for {longest:.2f} s of {spent[0]:.2f}"
