"""Outputs the binding allocates itself: their status words are cleared by the
call's own first kernel (SPIFFY_FRESH_STATUS), whatever the memory held."""
import pytest
import torch

from paper_2509_18085_b200 import spiffy
from paper_2509_18085_b200 import workloads as W
import gpu_util as G

pytestmark = pytest.mark.gpu


def poison():
    """Leaves set bits in the blocks the next small allocations come from."""
    blocks = [torch.full((n,), -1, dtype=torch.int32, device="cuda") for n in (1 << 20, 1 << 14, 1 << 10) for _ in range(4)]
    torch.cuda.synchronize()
    del blocks


@pytest.mark.parametrize("call", ["decide", "decide_walk", "lazy", "sampled", "walk", "draft", "lmhead"])
@pytest.mark.parametrize("bad_row", [False, True])
@pytest.mark.parametrize("N,L", [(3, 5), (18, 32)])  # fused tail; separate finalize and walk
def test_fresh_status_words_hold_this_call_only(call, bad_row, N, L):
    V = 1000
    cfg = W.Config("fresh", dtype="f32", vocab=V, rule=spiffy.RULE_TOPS, batch=3, n_nodes=N, block_len=L, prefix_len=0,
                   n_q_heads=1, n_kv_heads=1, head_dim=64)
    w = W.make(cfg, 5, attention=False)
    lg, tk, off, idx = (G.to_dev(a) for a in (w.logits, w.block_tokens, w.parent_off, w.parent_idx))
    masked = int((w.block_tokens[1, 0] == cfg.mask_id).nonzero()[0][0])
    if bad_row:
        lg[1, 0, masked, 17] = float("nan")
    args = (cfg.mask_id, cfg.rule)
    dec = spiffy.spiffy_unmask_decide(lg, tk, *args)
    poison()
    if call == "decide":
        status = spiffy.spiffy_unmask_decide(lg, tk, *args).dev_status
    elif call in ("decide_walk", "lazy"):
        d, wk = spiffy.spiffy_decide_walk(lg, tk, off, idx, *args, lazy=call == "lazy")
        status = d.dev_status
        assert wk.dev_status.tolist() == [0, 0, 0]
    elif call == "sampled":
        status = spiffy.spiffy_unmask_decide_sampled(lg, tk, *args, 1.0, 7).dev_status
    elif call == "draft":
        graph = spiffy.draft_graph([[(0, 0)], [(1, 0)]], [[1], []])
        d = spiffy.spiffy_draft_blocks(lg[:, 0].contiguous(), tk[:, 0].contiguous(), cfg.mask_id, graph, 2, 2, parent_cap=40)
        status = d.dev_status
        used = d.parent_off[:, -1].tolist()
        assert all(d.parent_idx[b, used[b]:].count_nonzero() == 0 for b in range(3))
    elif call == "lmhead":
        h = torch.randn((3, N, L, 128), device="cuda").to(torch.bfloat16)
        if bad_row:
            h[1, 0, masked, 3] = float("nan")
        status = spiffy.spiffy_lmhead_decide(h, torch.randn((V, 128), device="cuda").to(torch.bfloat16), tk, *args).dev_status
    else:
        if bad_row:
            off = off.clone()
            off[1, 1] = -5
        walk = spiffy.spiffy_accept_walk(tk, off, idx, dec.top_tok, dec.unmask_bits)
        assert walk.dev_status.tolist() == [0, spiffy.DEV_BADGRAPH if bad_row else 0, 0]
        return
    assert status.tolist() == [0, spiffy.DEV_NONFINITE if bad_row else 0, 0]
