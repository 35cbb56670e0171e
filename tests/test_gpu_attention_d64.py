"""Head dimension 64 in bf16 on the tensor cores (what SPIFFY_ATTN_AUTO takes),
at the edges of its tiles.  (Every one
of its routes: test_gpu_attention_routes.py.)"""
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
    (1, 8, 32, 512, 16, 16),                      # pairs of CTAs (as all above), as many key tiles as stages of the ring
    (1, 8, 32, 640, 16, 16),                      # ... one more
    (1, 9, 8, 1000, 3, 3),                        # clusters of eight
    (3, 9, 32, 300, 32, 32),                      # one M-tile per CTA, two rounds of CTAs
    (2, 9, 32, 300, 35, 35),                      # two M-tiles per CTA, the last one beyond the rows
    (1, 7, 32, 777, 32, 32),                      # 64 pairs
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


@pytest.mark.parametrize("B,N,L,P,Hq,Hkv", [(3, 5, 20, 777, 24, 8), (1, 8, 32, 512, 16, 16), (2, 9, 32, 4096, 32, 32),
                                            (1, 64, 4, 2048, 32, 8), (1, 3, 5, 50, 5, 5)])
@pytest.mark.parametrize("spread", [1.0, 4.0])
def test_no_less_precise_than_the_cuda_cores(B, N, L, P, Hq, Hkv, spread):
    """Probabilities enter the second product in two bf16 terms, right to 2^-16 of their value.  Both
    kernels' error is then the rounding of the result to bf16 (2^-9 of a value at most, 0.17 % in the
    2-norm): in quadrature the rest is 1e-4 of it.  One bf16 term would make the error a fifth larger."""
    g = torch.Generator(device="cuda").manual_seed(P)
    r = lambda *s: torch.randn(s, generator=g, device="cuda").to(torch.bfloat16)
    q, kp, vp, kb, vb = r(B, N, L, Hq, 64) * spread, r(B, P, Hkv, 64), r(B, P, Hkv, 64), r(B, N, L, Hkv, 64), r(B, N, L, Hkv, 64)
    want = float64_attention(q, kp, vp, kb, vb)
    err = {}
    for kernel in (spiffy.ATTN_AUTO, spiffy.ATTN_SIMT):
        out = spiffy.spiffy_graph_attention(q, kp, vp, kb, vb, kernel=kernel).double()
        err[kernel] = float((out - want).norm() / want.norm())
    print(err)
    assert err[spiffy.ATTN_AUTO] <= 1.005 * err[spiffy.ATTN_SIMT]


def float64_attention(q, kp, vp, kb, vb):
    (B, N, L, Hq, d), Hkv = q.shape, kp.shape[2]
    group = Hq // Hkv
    up = lambda t: t.double().repeat_interleave(group, dim=-2)
    out = torch.empty(q.shape, dtype=torch.float64, device=q.device)
    for b in range(B):
        kc, vc = up(kp[b]), up(vp[b])
        for n in range(N):
            k, v = torch.cat([kc, up(kb[b, n])]), torch.cat([vc, up(vb[b, n])])
            p = torch.softmax(torch.einsum("lhd,khd->hlk", q[b, n].double(), k) / d ** 0.5, -1)
            out[b, n] = torch.einsum("hlk,khd->lhd", p, v)
    return out
