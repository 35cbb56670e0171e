"""Every route of the tensor-core attention (attention_shapes.py): parity with the oracle, nothing written
beside the output, bit-identical reruns, waits that give up, and the layers of a model one behind the other."""
import numpy as np
import pytest
import torch

import oracle
from paper_2509_18085_b200 import spiffy
from paper_2509_18085_b200 import workloads as W
import gpu_util as G
from attention_shapes import CHAINS, GROWING, SHAPES
from test_gpu_canaries import Fenced

pytestmark = pytest.mark.gpu


def workload(shape, d, seed):
    return W.make(W.Config("route", *shape, d, "bf16", 16, 0), seed, decision=False)


def on_device(w):
    return [None if a is None or a.shape[1] == 0 else G.to_dev(a, torch.bfloat16)
            for a in (w.q, w.k_prefix, w.v_prefix, w.k_block, w.v_block)]


def check(w):
    """Output against the oracle, out of a buffer with guarded margins, twice the same bits.

    What an element may be off: bf16 rounds to 2^-8 of a value.  The result is rounded once; at head dimension 128
    so is each weight of the second product (2^-8 of the sum of the weighted |v|), at 64 its two terms keep 2^-16.
    A score is a sum of exact products in fp32 and is scaled in fp32, right to some 2^-21 of the largest |q| |k|
    / sqrt(d); as much is what a weight, its exponential, is off relatively, twice with the sum that divides it."""
    q, kp, vp, kb, vb = on_device(w)
    f = Fenced()
    out, status = f.tensor(tuple(q.shape), torch.bfloat16), f.tensor((1,), torch.int32)
    status.zero_()
    runs = []
    for _ in range(2):
        out.view(torch.uint8).fill_(0x5A)
        spiffy.spiffy_graph_attention(q, kp, vp, kb, vb, out=out, dev_status=status)
        f.check()
        runs.append(out.clone())
    assert torch.equal(runs[0].view(torch.int16), runs[1].view(torch.int16))
    assert int(status[0]) == 0
    got = out.float().cpu().numpy().astype(np.float64)
    want = oracle.graph_attention(w.q, w.k_prefix, w.v_prefix, w.k_block, w.v_block)
    weighted = oracle.graph_attention(w.q, w.k_prefix, np.abs(w.v_prefix), w.k_block, np.abs(w.v_block))
    d = w.q.shape[-1]
    norm = lambda *ts: max(float(np.sqrt((t.astype(np.float64) ** 2).sum(-1)).max(initial=0.0)) for t in ts)
    score = norm(w.q) * norm(w.k_prefix, w.k_block) / np.sqrt(d)
    bound = 2.0 ** -8 * np.abs(want) + ((2.0 ** -8 if d == 128 else 2.0 ** -15) + 2.0 ** -20 * score) * weighted
    assert np.all(np.abs(got - want) <= bound + 1e-6), float((np.abs(got - want) / bound).max())


@pytest.mark.parametrize("route,shape,d", SHAPES)
def test_parity_inside_the_buffers(route, shape, d):
    check(workload(shape, d, 23 + shape[3]))


@pytest.mark.parametrize("factor", [1.0, 10.0])
@pytest.mark.parametrize("route,shape,d", GROWING)
def test_maxima_that_grow_from_tile_to_tile(route, shape, d, factor):
    w = workload(shape, d, 3)
    w.q *= factor
    w.k_prefix *= (1.0 + np.arange(w.k_prefix.shape[1]) // 100 * 0.5)[None, :, None, None].astype(w.k_prefix.dtype)
    w.k_prefix[:, ::7] *= 2.0
    for a in ("q", "k_prefix"):
        setattr(w, a, W.round_to(getattr(w, a), "bf16"))
    check(w)


@pytest.mark.parametrize("route,shape,d", CHAINS)
def test_waits_that_may_not_poll_give_up(route, shape, d):
    w = workload(shape, d, 5)
    q, kp, vp, kb, vb = on_device(w)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    want = spiffy.spiffy_graph_attention(q, kp, vp, kb, vb, dev_status=status)
    torch.cuda.synchronize()
    assert int(status) == 0
    spiffy.set_wait_limits(mbarrier_polls=0)
    try:
        spiffy.spiffy_graph_attention(q, kp, vp, kb, vb, dev_status=status)
        torch.cuda.synchronize()
    finally:
        spiffy.set_wait_limits()
    assert int(status) == spiffy.DEV_TIMEOUT
    status.zero_()
    again = spiffy.spiffy_graph_attention(q, kp, vp, kb, vb, dev_status=status)
    torch.cuda.synchronize()
    assert int(status) == 0 and torch.equal(again, want)


@pytest.mark.parametrize("route,shape,d", CHAINS)
def test_layers_that_let_the_next_one_begin_early(route, shape, d):
    """SPIFFY_ATTN_EARLY_DEPENDENTS: each layer's queries are the one before's output, the first one's are written
    just ahead of it, and a decision and a walk follow.  Bit for bit what the calls give without the flag, each
    waited for."""
    w = workload(shape, d, 7)
    q, kp, vp, kb, vb = on_device(w)
    B, N, L = shape[:3]
    vocab = 1000
    tokens = torch.full((B, N, min(L, 64)), vocab - 1, dtype=torch.int32, device="cuda")
    off = torch.zeros((B, N + 1), dtype=torch.int32, device="cuda")
    idx = torch.zeros((B, 1), dtype=torch.int32, device="cuda")
    g = torch.Generator(device="cuda").manual_seed(1)
    logits = torch.randn((B, N, min(L, 64), vocab), generator=g, device="cuda").to(torch.bfloat16)
    inputs = [q, torch.randn(q.shape, generator=g, device="cuda").to(torch.bfloat16)]
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    layers = 5

    def run(x, flags, between):
        outs = [torch.full_like(q, float("nan")) for _ in range(layers + 1)]
        torch.cuda.synchronize()
        outs[0].copy_(x)
        for i in range(layers):
            spiffy.spiffy_graph_attention(outs[i], kp, vp, kb, vb, out=outs[i + 1], kernel=spiffy.ATTN_AUTO | flags,
                                          dev_status=status)
            between()
        dec, walk = spiffy.spiffy_decide_walk(logits, tokens, off, idx, vocab - 1, spiffy.RULE_TOPS)
        torch.cuda.synchronize()
        return outs, dec, walk

    for x in inputs:
        outs, dec, walk = run(x, 0, torch.cuda.synchronize)
        for _ in range(8):
            outs2, dec2, walk2 = run(x, spiffy.ATTN_EARLY_DEPENDENTS, lambda: None)
            for a, b in zip(outs, outs2):
                assert torch.equal(a.view(torch.int16), b.view(torch.int16))
            G.assert_same_bits(dec, walk, dec2, walk2)
    assert int(status) == 0
    assert not any(torch.isnan(o).any() for o in outs)
