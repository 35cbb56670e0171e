"""The CUDA-core attention kernel at the edges of its row tiles (16, 32, 64),
key tiles (64) and key slices (clusters of 1 to 8)."""
import numpy as np
import pytest

import oracle
from paper_2509_18085_b200 import spiffy
from paper_2509_18085_b200 import workloads as W
import gpu_util as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("B,N,L,P,Hq,Hkv", [
    (1, 1, 1, 0, 1, 1), (1, 1, 1, 1, 1, 1),
    (1, 2, 9, 63, 4, 4), (1, 2, 9, 64, 4, 4), (1, 3, 11, 65, 4, 4),  # 16-row tiles, a partial one
    (2, 2, 4, 3249, 24, 8),                                          # few rows, eight slices
    (1, 1, 37, 200, 40, 40),                                         # 32-row tiles or 64, two slices
    (1, 13, 31, 56, 32, 8),                                          # many rows, one slice
    (2, 2, 64, 129, 3, 3), (1, 2, 3, 20, 200, 1)])                   # the longest block; 200 heads on one kv head
def test_parity(B, N, L, P, Hq, Hkv, d, dtype):
    cfg = W.Config("simt", B, N, L, P, Hq, Hkv, d, dtype, 16, 0)
    w = W.make(cfg, 3 + P, decision=False)
    got = G.gpu_attention(w, spiffy.ATTN_SIMT)
    want = oracle.graph_attention(w.q, w.k_prefix, w.v_prefix, w.k_block, w.v_block)
    assert np.max(np.abs(got - want)) <= (2e-6 if dtype == "f32" else G.TOL["bf16"]) * (1 + np.max(np.abs(want)))
