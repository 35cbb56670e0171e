"""How the tensor-core attention shares out its key tiles: few of them among the softmax
warpgroups of a pair of CTAs, clusters of 8 CTAs, one M-tile per CTA, two, a last round in a
launch of its own.  (Clusters of 2 and 4, and each route's edges: test_gpu_attention_routes.py.)"""
import numpy as np
import pytest

import oracle
from paper_2509_18085_b200 import spiffy
from paper_2509_18085_b200 import workloads as W
import gpu_util as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,N,L,P,Hq,Hkv", [
    # pairs: one key tile, so that three of the four warpgroups have none ...
    (1, 2, 16, 0, 2, 2),
    (1, 4, 32, 100, 4, 4),        # ... two
    (1, 4, 32, 128 * 2, 64, 64),  # ... three
    (1, 1, 7, 128 * 6, 2, 1),     # ... seven, eight, nine: two turns, and a third for one
    (1, 1, 7, 128 * 7, 2, 1), (1, 1, 7, 128 * 7 + 1, 2, 1),
    (1, 6, 32, 2562, 8, 1),       # a cluster of 8
    (1, 2, 32, 1746, 28, 4),      # pairs, the ring of stages three times round
    (1, 4, 32, 900, 30, 30),      # ... 60 CTAs of them
    (1, 7, 32, 777, 32, 32),      # ... 128
    (2, 9, 32, 500, 40, 40),      # one M-tile per CTA, two rounds of CTAs
    (4, 32, 32, 140, 16, 8),      # two M-tiles per CTA
    (2, 9, 32, 300, 35, 35)])     # ... an odd number of them: the last CTA's second one is empty
def test_parity(B, N, L, P, Hq, Hkv):
    cfg = W.Config("splits", B, N, L, P, Hq, Hkv, 128, "bf16", 16, 0)
    w = W.make(cfg, 11 + P, decision=False)
    got = G.gpu_attention(w, spiffy.ATTN_TCGEN05)
    want = oracle.graph_attention(w.q, w.k_prefix, w.v_prefix, w.k_block, w.v_block)
    assert np.max(np.abs(got - want)) <= G.TOL["bf16"]
    assert np.sqrt(np.mean((got - want) ** 2)) < 4e-3
    assert np.array_equal(got, G.gpu_attention(w, spiffy.ATTN_TCGEN05))


def test_late_maximum_in_another_slice():
    """The largest scores sit in the last slice of a cluster, and in tiles of one
    warpgroup only: partials with very different reference maxima are merged."""
    cfg = W.Config("splits", 1, 2, 16, 128 * 16, 2, 1, 128, "bf16", 16, 0)
    w = W.make(cfg, 5, decision=False)
    w.q *= 6.0
    w.k_prefix[:, 128 * 14:128 * 15] *= 3.0
    for a in ("q", "k_prefix"):
        setattr(w, a, W.round_to(getattr(w, a), "bf16"))
    got = G.gpu_attention(w, spiffy.ATTN_TCGEN05)
    want = oracle.graph_attention(w.q, w.k_prefix, w.v_prefix, w.k_block, w.v_block)
    assert np.all(np.isfinite(got)) and np.max(np.abs(got - want)) <= G.TOL["bf16"]


@pytest.mark.parametrize("B,N,L,P,Hq,Hkv", [
    (5, 8, 25, 100, 64, 64),    # 320 CTAs of two M-tiles: 24 of them, beyond two rounds, by pairs of blocks
    (4, 7, 20, 40, 89, 89),     # 356: 60 of them with one M-tile per block
    (2, 10, 30, 50, 90, 90),    # ... three M-tiles a head: every fourth block of the second launch has none
    (3, 5, 60, 20, 330, 110)])  # one launch after all: groups of three query heads, eight rounds and most of a ninth
def test_last_round_in_a_launch_of_its_own(B, N, L, P, Hq, Hkv):
    cfg = W.Config("splits", B, N, L, P, Hq, Hkv, 128, "bf16", 16, 0)
    w = W.make(cfg, 17 + P, decision=False)
    got = G.gpu_attention(w, spiffy.ATTN_TCGEN05)
    want = oracle.graph_attention(w.q, w.k_prefix, w.v_prefix, w.k_block, w.v_block)
    assert np.max(np.abs(got - want)) <= G.TOL["bf16"]
    assert np.sqrt(np.mean((got - want) ** 2)) < 4e-3
    assert np.array_equal(got, G.gpu_attention(w, spiffy.ATTN_TCGEN05))
