"""spiffy_lmhead_decide at the numbers of masked positions where its tiles, ring
and accumulators change: steps of 16 and 32, 128 (two accumulator pairs below),
256 (passes), and at vocabularies whose shares end inside a tile."""
import numpy as np
import pytest
import torch

import oracle
from paper_2509_18085_b200 import spiffy

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count,V,H", [(0, 500, 128), (1, 31, 128), (15, 33, 256), (16, 4736, 128), (17, 4737, 640),
                                       (33, 40000, 128), (127, 9000, 256), (128, 9001, 256), (129, 9002, 256),
                                       (255, 38000, 384), (256, 1000, 128), (257, 5000, 128), (600, 300, 256), (166, 80000, 128),
                                       (300, 45000, 128)])
def test_every_count_of_masked_positions(count, V, H):
    g = torch.Generator().manual_seed(count + V)
    L = 40
    N = (max(count, 1) + 20 + L - 1) // L
    hs = torch.randn((1, N, L, H), generator=g).to(torch.bfloat16)
    w = (torch.randn((V, H), generator=g) * (2.0 / H ** 0.5)).to(torch.bfloat16)
    tokens = torch.full((N * L,), 3, dtype=torch.int32)
    tokens[torch.randperm(N * L, generator=g)[:count]] = -7
    tokens = tokens.reshape(1, N, L)
    dec = spiffy.spiffy_lmhead_decide(hs.cuda(), w.cuda(), tokens.cuda(), -7, spiffy.RULE_THRESHOLD, 1, 0.02)
    again = spiffy.spiffy_lmhead_decide(hs.cuda(), w.cuda(), tokens.cuda(), -7, spiffy.RULE_THRESHOLD, 1, 0.02)
    torch.cuda.synchronize()
    logits = (hs.double().reshape(-1, H) @ w.double().T).reshape(1, N, L, V).numpy()
    o = oracle.unmask_decide(logits.astype(np.float32), tokens.numpy(), -7, spiffy.RULE_THRESHOLD, 1, 0.02)
    srt = np.sort(logits, axis=-1)
    m = tokens.numpy() == -7
    sure = m & (srt[..., -1] - srt[..., -2] > 1e-3)
    tok = dec.top_tok.cpu().numpy()
    assert np.array_equal(tok[sure], o.top_tok[sure]) and np.array_equal(tok[~m], tokens.numpy()[~m])
    np.testing.assert_allclose(dec.conf.cpu().numpy()[m], o.conf[m], atol=1e-4)
    assert torch.equal(dec.conf.view(torch.int32), again.conf.view(torch.int32)) and torch.equal(dec.top_tok, again.top_tok)
    assert int(dec.dev_status.sum()) == 0
