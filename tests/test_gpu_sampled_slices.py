"""The sampled decision on either side of a vocabulary of one slice (one kernel
reduces and draws below, two above), at ragged vocabularies in padded rows, and
the status word with and without arbitrary contents."""
import numpy as np
import pytest
import torch

from oracle import sampling as S
from paper_2509_18085_b200 import spiffy
import gpu_util as G
from test_gpu_sampled import CDF_GAP, SLICE_GAP, case

pytestmark = pytest.mark.gpu


def padded(logits, dtype):
    t = torch.from_numpy(logits).to(torch.bfloat16 if dtype == "bf16" else torch.float32)
    V = t.shape[-1]
    room = torch.full((*t.shape[:-1], (V + 7) // 8 * 8), 40.0, dtype=t.dtype, device="cuda")
    room[..., :V] = t.cuda()
    return room[..., :V]


@pytest.mark.parametrize("dtype,V,N,L", [("bf16", 3, 1, 1), ("bf16", 1021, 40, 3), ("bf16", 8191, 3, 33),
                                         ("bf16", 8192, 2, 64), ("bf16", 8193, 2, 9), ("f32", 4093, 17, 4),
                                         ("f32", 4096, 2, 5), ("f32", 4097, 2, 5)])
def test_around_one_slice(dtype, V, N, L):
    logits, tokens, mask = case(V, 2, N, L, V, dtype)
    dl, dt = padded(logits, dtype), G.to_dev(tokens)
    dec = spiffy.spiffy_unmask_decide_sampled(dl, dt, mask, spiffy.RULE_TOPS, 0.8, 77, 2, 0.0)
    width = spiffy.spiffy_sampled_slice_width(spiffy.decide_desc(dl, dt, mask, spiffy.RULE_TOPS, 2, 0.0))
    o = S.sampled_decide(logits, tokens, mask, spiffy.RULE_TOPS, 2, 0.0, 0.8, 77, width)
    sure = (o.slice_gap > SLICE_GAP) & (o.cdf_gap > CDF_GAP)
    assert sure.mean() > 0.97
    assert np.array_equal(dec.top_tok.cpu().numpy()[sure], o.top_tok[sure])
    ok = sure & (tokens == mask)
    np.testing.assert_allclose(dec.conf.cpu().numpy()[ok], o.conf[ok], atol=1e-4)
    node_ok = sure.all(axis=2) & (o.margin > 1e-3)
    assert np.array_equal(G.bits_np(dec.unmask_bits)[node_ok], o.unmask_bits[node_ok])
    assert np.array_equal(dec.n_unmask.cpu().numpy()[node_ok], o.n_unmask[node_ok])
    assert int(dec.dev_status.abs().sum()) == 0


@pytest.mark.parametrize("V", [1000, 9000])
def test_status_is_ored_into_what_the_caller_left(V):
    logits, tokens, mask = case(3, 2, 2, 4, V, "f32")
    logits[1, 1, 0] = np.nan
    dl, dt = G.to_dev(logits), G.to_dev(tokens)
    fresh = spiffy.spiffy_unmask_decide_sampled(dl, dt, mask, spiffy.RULE_TOPS, 1.0, 5, 1, 0.0)
    assert fresh.dev_status.tolist() == [0, spiffy.DEV_NONFINITE]
    fresh.dev_status.fill_(1 << 20)
    spiffy.spiffy_unmask_decide_sampled(dl, dt, mask, spiffy.RULE_TOPS, 1.0, 5, 1, 0.0, out=fresh)
    assert fresh.dev_status.tolist() == [1 << 20, 1 << 20 | spiffy.DEV_NONFINITE]
