"""VerifyStep.run, where decision and attention run side by side, against the
same calls one after the other: bit-identical on every path the two kernels
have (tail in one CTA, separate finalize and walk, both attention kernels, one
and several rounds of CTAs), many steps back to back on alternating inputs."""
import dataclasses

import pytest
import torch

from paper_2509_18085_b200 import spiffy
from paper_2509_18085_b200 import workloads as W
from paper_2509_18085_b200.step import VerifyStep, inputs_from_workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,N,L,P,Hq,Hkv,d,V,dtype", [
    (1, 2, 4, 0, 4, 4, 128, 1000, "bf16"),      # nothing to share the machine with
    (3, 24, 4, 764, 24, 8, 128, 4000, "bf16"),  # one nearly full round of clusters
    (1, 54, 32, 300, 28, 4, 64, 4072, "bf16"),  # more than 512 rows: finalize and walk kernels
    (2, 16, 32, 2000, 32, 32, 128, 8192, "bf16"),  # several rounds
    # a call of two launches, the second by pairs and by one M-tile per block; beside the fused tail and not
    (5, 8, 32, 256, 32, 32, 128, 1000, "bf16"), (1, 18, 60, 100, 150, 50, 128, 1000, "bf16"),
    (2, 3, 32, 500, 5, 5, 128, 2864, "f32"),
    # fp32: the decision in one launch, up to 64 slices a sequence and 8 sequences, and just beyond
    (1, 1, 1, 60, 1, 1, 64, 52, "f32"), (8, 4, 16, 60, 4, 4, 64, 1000, "f32"), (9, 4, 16, 60, 4, 4, 64, 1000, "f32"),
    (1, 3, 21, 60, 4, 4, 64, 4096, "f32"), (1, 1, 64, 60, 4, 4, 64, 4096, "f32"), (2, 1, 64, 60, 4, 4, 64, 4100, "f32"),
    (3, 4, 4, 60, 4, 4, 64, 16384, "f32"), (1, 64, 1, 60, 4, 4, 64, 300, "f32"), (1, 65, 1, 60, 4, 4, 64, 300, "f32"),
])
def test_same_bits_as_one_after_the_other(B, N, L, P, Hq, Hkv, d, V, dtype):
    cfg = W.Config("t", B, N, L, P, Hq, Hkv, d, dtype, V, spiffy.RULE_THRESHOLD)
    step, apart = VerifyStep(cfg), VerifyStep(cfg)
    xs = [inputs_from_workload(W.make(cfg, s)) for s in (1, 2, 3)]
    want = []
    for x in xs:
        apart.attention(x)
        apart.decide_accept(x)
        want.append(_results(apart))
    for i in range(30):
        step.run(xs[i % 3])
        if i % 7 == 0 or i > 26:
            for a, b in zip(_results(step), want[i % 3]):
                assert torch.equal(a, b)


@pytest.mark.parametrize("N,V,dtype", [(16, 4000, "bf16"), (16, 70000, "bf16"), (17, 4000, "bf16"),
                                       (16, 4000, "f32"), (16, 40000, "f32"), (17, 4000, "f32")])
def test_late_in_a_block(N, V, dtype):
    """Most rows unmasked, the last one among them: the blocks of the reduce that end at once, and the one that
    waits for the kernel before, on both routes of the decision."""
    cfg = W.Config("t", 1, N, 32, 300, 8, 4, 64, dtype, V, spiffy.RULE_THRESHOLD)
    step, apart = VerifyStep(cfg), VerifyStep(cfg)
    x = inputs_from_workload(W.make(cfg, 4))
    for masked in (0, 3, 40):
        x.block_tokens.fill_(7)
        at = torch.randperm(N * 31, generator=torch.Generator().manual_seed(masked))[:masked].cuda()
        x.block_tokens[0, at // 31, at % 31] = cfg.mask_id  # the last position of every node stays
        apart.attention(x)
        apart.decide_accept(x)
        want = _results(apart)
        for _ in range(5):
            step.run(x)
            for a, b in zip(_results(step), want):
                assert torch.equal(a, b)


@pytest.mark.parametrize("N,L", [(4, 8), (1, 64), (9, 16)])  # in one launch, in two
def test_results_may_lie_where_the_attention_reads(N, L):
    """SPIFFY_INDEPENDENT is about the decision's inputs: its results may replace keys that the attention in front,
    which takes far longer, has yet to read."""
    cfg = W.Config("t", 2, N, L, 6000, 8, 8, 128, "f32", 1000, spiffy.RULE_THRESHOLD)
    x, apart = inputs_from_workload(W.make(cfg, 8)), VerifyStep(cfg)
    apart.attention(x)
    apart.decide_accept(x)
    want, keys, step = _results(apart), x.k_prefix.clone(), VerifyStep(cfg)
    room, at = x.k_prefix.view(-1), x.k_prefix.numel()

    def moved(t):  # from the last keys backwards
        nonlocal at
        at -= -(-t.numel() * t.element_size() // 64) * 16
        return room[at:at + t.numel() * t.element_size() // 4].view(t.dtype).view(t.shape)

    for results in (step.decision, step.walk):
        for f in dataclasses.fields(results):
            if f.name != "dev_status":  # OR-ed into what is there
                setattr(results, f.name, moved(getattr(results, f.name)))
    for _ in range(3):
        x.k_prefix.copy_(keys)
        step.run(x)
        for a, b in zip(_results(step), want):
            assert torch.equal(a, b)


@pytest.mark.parametrize("flags", [spiffy.INDEPENDENT, spiffy.INDEPENDENT | spiffy.INDEPENDENT_NEXT])
@pytest.mark.parametrize("rule,S", [(spiffy.RULE_TOPS, 1), (spiffy.RULE_TOPS, 3), (spiffy.RULE_TOPS, 9), (spiffy.RULE_THRESHOLD, 1)])
@pytest.mark.parametrize("B,N,L,V,dtype", [(8, 4, 16, 1000, "bf16"), (3, 8, 4, 16384, "bf16"), (2, 4, 8, 8000, "f32"),
                                           (2, 64, 1, 300, "f32"), (1, 2, 32, 8192, "bf16"), (5, 3, 5, 12004, "f32")])
def test_one_launch_with_odd_inputs(B, N, L, V, dtype, rule, S, flags):
    """Behind an attention on the CUDA cores: rows that hold a NaN, an infinity or nothing but -inf, nodes with all
    positions unmasked, malformed lists, status words that are OR-ed into or arrive with anything."""
    cfg = W.Config("t", B, N, L, 40, 4, 4, 64, dtype, V, rule, S)
    x = inputs_from_workload(W.make(cfg, 11))
    x.logits[0, 0, L - 1, 1::2] = float("-inf")  # still a distribution
    x.block_tokens[:, N // 2] = 5
    spoiled = [0] * B
    if B > 1:
        x.logits[1, 0, 0, V // 2], spoiled[1] = float("nan"), spiffy.DEV_NONFINITE
        x.block_tokens[1, 0, 0] = cfg.mask_id
    if B > 2:
        x.logits[2, N - 1, L - 1], spoiled[2] = float("-inf"), spiffy.DEV_NONFINITE
        x.logits[2, 0, 0, 3] = float("inf")
        x.block_tokens[2, N - 1, L - 1] = x.block_tokens[2, 0, 0] = cfg.mask_id
    whole = torch.tensor([s == 0 for s in spoiled], device="cuda")
    for lists in ("good", "entry", "offset"):
        off, idx, bad = x.parent_off.clone(), x.parent_idx.clone(), 0
        if lists != "good":
            bad = spiffy.DEV_BADGRAPH
            if lists == "entry":
                off[0, 1:], idx[0, 0] = 1, N  # a node's one parent is a node that is not there
                off[0, 1] = 0
            else:
                off[0, N - 1] = -3
        args = (cfg.mask_id, cfg.rule, cfg.top_s, cfg.threshold)
        dec = spiffy.spiffy_unmask_decide(x.logits, x.block_tokens, *args)
        walk = spiffy.spiffy_accept_walk(x.block_tokens, off, idx, dec.top_tok, dec.unmask_bits)
        assert dec.dev_status.tolist() == spoiled and walk.dev_status.tolist() == [bad] + [0] * (B - 1)
        for kept in (True, False):
            d, w = VerifyStep(cfg, attn_kernel=spiffy.ATTN_SIMT).decision, VerifyStep(cfg, attn_kernel=spiffy.ATTN_SIMT).walk
            d.dev_status.fill_(64)
            w.dev_status.fill_(32)
            spiffy.spiffy_graph_attention(x.q, x.k_prefix, x.v_prefix, x.k_block, x.v_block, kernel=spiffy.ATTN_SIMT)
            before = spiffy.launch_count()
            got_d, got_w = spiffy.spiffy_decide_walk(x.logits, x.block_tokens, off, idx, *args, decision=d if kept else None,
                                                     walk=w if kept else None, flags=flags)
            assert spiffy.launch_count() - before == 1
            assert got_d.dev_status.tolist() == [s | (64 if kept else 0) for s in spoiled]
            assert got_w.dev_status.tolist() == [s | (32 if kept else 0) for s in [bad] + [0] * (B - 1)]
            for a, b in zip(_fields(got_d)[:-1] + _fields(got_w)[:-1], _fields(dec)[:-1] + _fields(walk)[:-1]):
                assert torch.equal(a[whole].view(torch.uint8), b[whole].view(torch.uint8))


def _results(s):
    out = [s.attn_out, s.attn_status] + list(_fields(s.decision)) + list(_fields(s.walk))
    return [t.clone().view(torch.uint8) for t in out]


def _fields(x):
    return [getattr(x, f.name) for f in dataclasses.fields(x)] if dataclasses.is_dataclass(x) else list(x)


@pytest.mark.parametrize("pinned", ["all", "lists not", "logits not", "verdict not"])
@pytest.mark.parametrize("N,L,Hq,Hkv,d,dtype", [(5, 8, 4, 4, 128, "bf16"), (40, 20, 8, 2, 64, "bf16"), (3, 5, 2, 2, 64, "f32")])
def test_host_step_from_pinned_and_pageable_arrays(pinned, N, L, Hq, Hkv, d, dtype):
    cfg = W.Config("t", 2, N, L, 70, Hq, Hkv, d, dtype, 1000, spiffy.RULE_THRESHOLD)
    w = W.make(cfg, 5)
    step = VerifyStep(cfg)
    step.run(inputs_from_workload(w))
    want = [t.cpu() for t in (step.walk.accepted_node, step.walk.n_accepted, step.walk.path, step.walk.next_block)]
    host = inputs_from_workload(w, device="cpu", pin=True)
    if pinned == "lists not":
        host.parent_off, host.parent_idx = host.parent_off.clone(), host.parent_idx.clone()
    if pinned == "logits not":
        host.logits = host.logits.clone()
    for i in range(3):
        got = step.run_host(host)
        if pinned == "verdict not" and i == 0:
            step.host_verdict = tuple(torch.full_like(t, 77) for t in step.host_verdict)
            continue
        for a, b in zip(step.host_verdict, want):
            assert torch.equal(a, b)
        assert int(step.host_verdict[4].abs().sum()) == 0
        for t in step.host_verdict:
            t.fill_(77)
