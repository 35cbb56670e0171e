"""Attention by pairs of thread blocks: the sizes at which their division of labour has edges."""
import numpy as np
import pytest
import torch

import oracle
from oracle import full_mask
from paper_2509_18085_b200 import spiffy
from paper_2509_18085_b200 import workloads as W
import gpu_util as G

pytestmark = pytest.mark.gpu


def check(cfg, seed, scale=None):
    w = W.make(cfg, seed, decision=False)
    if scale:
        scale(w)
    kernel = spiffy.ATTN_TCGEN05 if cfg.head_dim == 128 else spiffy.ATTN_AUTO
    got = G.gpu_attention(w, kernel)
    want = oracle.graph_attention(w.q, w.k_prefix, w.v_prefix, w.k_block, w.v_block)
    assert np.max(np.abs(got - want)) <= G.TOL["bf16"]
    assert np.sqrt(np.mean((got - want) ** 2)) < 4e-3
    assert np.array_equal(got, G.gpu_attention(w, kernel))


@pytest.mark.parametrize("d", [128, 64])
@pytest.mark.parametrize("B,N,L,P,Hq,Hkv", [
    (1, 1, 4, 0, 1, 1),            # one key tile: three warpgroups without any, the second block without rows
    (1, 2, 32, 0, 2, 2), (1, 2, 33, 60, 2, 2),   # 64 rows, and two more in the second block
    (1, 4, 32, 128 * 3, 3, 3),     # as many key tiles as warpgroups
    (1, 5, 32, 128 * 3 + 1, 3, 3),  # one more; the last pair has one block's rows
    # as many as the ring has stages, one more (at head dimension 64 that many already, then a cluster)
    (2, 4, 32, 128 * 5, 3, 3), (2, 4, 32, 128 * 6, 3, 3),
    (1, 3, 17, 128 * 12 - 3, 28, 4),  # long enough for a cluster of eight instead
    (1, 9, 34, 128 * 12 - 3, 28, 4),  # the ring several times round, groups of 7: 63 rows of 64
    (1, 3, 5, 190, 64, 1), (1, 7, 3, 300, 66, 2),   # one position a block; groups of 33
    (1, 1, 200, 65, 2, 1),         # block keys over two key tiles
    (3, 4, 9, 449, 10, 2), (1, 9, 16, 1, 24, 8), (4, 2, 31, 127, 12, 4)])
def test_parity(B, N, L, P, Hq, Hkv, d):
    check(W.Config("pair", B, N, L, P, Hq, Hkv, d, "bf16", 16, 0), 100 + P)


@pytest.mark.parametrize("d", [128, 64])
@pytest.mark.parametrize("factor", [3.0, 40.0])
def test_maxima_that_grow_from_tile_to_tile(factor, d):
    """Accumulators are rescaled, in some rows by the other half's maximum alone.  (Head dimension 64: this
    shape goes to a cluster of eight; the pair's is in test_gpu_attention_routes.py.)"""
    def scale(w):
        w.q *= factor / 3.0
        w.k_prefix *= (1.0 + np.arange(w.k_prefix.shape[1]) // 100 * 0.5)[None, :, None, None].astype(w.k_prefix.dtype)
        w.k_prefix[:, ::7] *= 2.0
        for a in ("q", "k_prefix"):
            setattr(w, a, W.round_to(getattr(w, a), "bf16"))
    check(W.Config("pair", 1, 4, 20, 128 * 9 + 5, 6, 3, d, "bf16", 16, 0), 3, scale)


def test_two_problems_in_one_launch():
    g = torch.Generator().manual_seed(9)
    B, N, L, P, S, Hq, Hkv, d = 2, 3, 20, 333, 45, 6, 3, 128
    r = lambda *s: torch.randn(s, generator=g).to(torch.bfloat16)
    q, qs, kp, vp, ks, vs, kb, vb = (r(B, N, L, Hq, d), r(B, S, Hq, d), r(B, P, Hkv, d), r(B, P, Hkv, d), r(B, S, Hkv, d),
                                     r(B, S, Hkv, d), r(B, N, L, Hkv, d), r(B, N, L, Hkv, d))
    out, out_s = spiffy.spiffy_full_sequence_attention(*(t.cuda() for t in (q, qs, kp, vp, ks, vs, kb, vb)))
    want, want_s = full_mask.full_sequence_attention(*(t.float().numpy() for t in (q, qs, kp, vp, ks, vs, kb, vb)))
    assert np.max(np.abs(out.float().cpu().numpy() - want)) <= G.TOL["bf16"]
    assert np.max(np.abs(out_s.float().cpu().numpy() - want_s)) <= G.TOL["bf16"]
