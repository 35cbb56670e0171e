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
    assert longest < 0.5 * spent[0], f"another thread stood still for {longest:.2f} s of {spent[0]:.2f}"


@pytest.mark.parametrize("call", ["decide", "decide_walk", "lazy", "sampled", "walk", "draft", "lmhead", "attention"])
def test_what_a_call_allocates_belongs_to_its_stream(call):
    """With `stream=` naming another than the current stream, memory of the call that has gone back to
    the allocator is not handed to work of the current stream while the call has yet to use it, and
    results do not land in memory that work of the current stream still uses."""
    cfg, (lg, tk, off, idx) = small(B=2, N=4, L=8, V=20000)
    args = (cfg.mask_id, cfg.rule)
    graph = spiffy.draft_graph([[(0, 0)], [(1, 0)]], [[1], []])
    h, w = (torch.randn(s, device="cuda").to(torch.bfloat16) for s in ((2, 4, 8, 128), (20000, 128)))
    first, block0 = lg[:, 0].contiguous(), tk[:, 0].contiguous()
    q, kv = (torch.randn((2, n, 8, 4, 64), device="cuda").to(torch.bfloat16) for n in (4, 4))
    dec = spiffy.spiffy_unmask_decide(lg, tk, *args)

    def run(stream=None):
        if call == "decide":
            r = [spiffy.spiffy_unmask_decide(lg, tk, *args, stream=stream)]
        elif call in ("decide_walk", "lazy"):
            r = spiffy.spiffy_decide_walk(lg, tk, off, idx, *args, stream=stream, lazy=call == "lazy")
        elif call == "sampled":
            r = [spiffy.spiffy_unmask_decide_sampled(lg, tk, *args, 0.8, 7, stream=stream)]
        elif call == "walk":
            r = [spiffy.spiffy_accept_walk(tk, off, idx, dec.top_tok, dec.unmask_bits, stream=stream)]
        elif call == "draft":
            r = [spiffy.spiffy_draft_blocks(first, block0, cfg.mask_id, graph, 2, 2, stream=stream)]
        elif call == "lmhead":
            r = [spiffy.spiffy_lmhead_decide(h, w, tk, *args, stream=stream)]
        else:
            return [spiffy.spiffy_graph_attention(q, None, None, kv, kv, stream=stream)]
        return [t for part in r for t in vars(part).values()]

    lazy_holes = {0, 1, 2}  # conf, top_tok, unmask_bits off the path are left as they were
    want = [t.clone() for t in run()]
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        torch.cuda._sleep(100_000_000)  # the call's kernels come some 50 ms after it returns
    got = run(side)
    # the current stream takes and fills whatever the call has given back by now
    mine = [torch.full((n,), 0x55, dtype=torch.uint8, device="cuda") for n in (1 << 9, 1 << 11, 1 << 13, 1 << 15) for _ in range(8)]
    torch.cuda.current_stream().synchronize()
    torch.cuda.synchronize()
    for i, (a, b) in enumerate(zip(got, want)):
        if call != "lazy" or i not in lazy_holes:
            assert torch.equal(a.view(torch.uint8), b.view(torch.uint8)), i
    for t in mine:
        assert int((t != 0x55).sum()) == 0
