"""Head dimension 64 in bf16 on the tensor cores (what SPIFFY_ATTN_AUTO takes),
at the edges of its tiles and on each of its routes."""
import numpy as np
import pytest
import torch

import oracle
from paper_2509_18085_b200 import spiffy
from paper_2509_18085_b200 import workloads as W
import gpu_util as G

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,N,L,P,Hq,Hkv", [
    (1, 1, 1, 1, 1, 1), (1, 2, 5, 0, 2, 1),       # the smallest; block keys only
    (1, 3, 7, 127, 16, 16), (1, 3, 7, 129, 16, 16),  # context one short of / one past a key tile
    (1, 8, 32, 512, 16, 16),                      # cluster pairs, odd number of key tiles
    (1, 8, 32, 640, 16, 16),                      # cluster pairs, even
    (1, 9, 8, 1000, 3, 3),                        # many slices through the workspace
    (3, 9, 32, 300, 32, 32),                      # two M-tiles per CTA, the second one partly beyond the rows
    (2, 4, 12, 129, 28, 4),                       # grouped heads: M-tiles of 126 rows
    (1, 2, 3, 20, 128, 1),                        # one position per M-tile
    (1, 1, 64, 2000, 4, 2)])
def test_parity(B, N, L, P, Hq, Hkv):
    cfg = W.Config("d64", B, N, L, P, Hq, Hkv, 64, "bf16", 16, 0)
    w = W.make(cfg, 7 + P, decision=False)
    got = G.gpu_attention(w)
    want = oracle.graph_attention(w.q, w.k_prefix, w.v_prefix, w.k_block, w.v_block)
    assert np.max(np.abs(got - want)) <= G.TOL["bf16"]
    assert np.sqrt(np.mean((got - want) ** 2)) < 4e-3


def test_reruns_are_bit_identical_and_the_kernel_is_the_tensor_core_one():
    cfg = W.Config("d64", 1, 8, 32, 512, 16, 16, 64, "bf16", 16, 0)
    w = W.make(cfg, 3, decision=False)
    a, b = G.gpu_attention(w), G.gpu_attention(w)
    assert np.array_equal(a, b)
    # a tensor-core wait that may not poll gives up; the CUDA-core kernel would not notice
    q, kp, vp, kb, vb = (G.to_dev(x, torch.bfloat16) for x in (w.q, w.k_prefix, w.v_prefix, w.k_block, w.v_block))
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    spiffy.set_wait_limits(mbarrier_polls=0)
    try:
        spiffy.spiffy_graph_attention(q, kp, vp, kb, vb, dev_status=status)
        torch.cuda.synchronize()
    finally:
        spiffy.set_wait_limits()
    assert int(status[0]) == spiffy.DEV_TIMEOUT
