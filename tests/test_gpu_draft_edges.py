"""Drafting around the 64 formulas whose subset relation is tabulated, with
every buildable formula kept, and top-k lists that come from one thread, one
vector or the ragged tail of a slice, with ties between token ids."""
import numpy as np
import pytest
import torch

from oracle import drafting
from paper_2509_18085_b200 import spiffy
import gpu_util as G
from test_gpu_draft import assert_parity, run_both

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D", [1, 63, 64, 65, 130])
def test_subset_relation_of_many_formulas(D):
    r = np.random.default_rng(D)
    pool = [(i, j) for i in range(9) for j in range(3)]
    formulas, seen = [], set()
    while len(formulas) < D:
        f = [pool[k] for k in sorted(r.choice(len(pool), size=r.integers(1, 4), replace=False))]
        if len({i for i, _ in f}) == len(f) and tuple(f) not in seen:
            seen.add(tuple(f))
            formulas.append(f)
    formulas.sort(key=len)
    children = [[int(x) for x in r.choice(D, size=min(2, D), replace=False)] for _ in range(D)]
    logits = (r.standard_normal((2, 10, 500)) * 3).astype(np.float32)
    state = np.full((2, 10), 499, dtype=np.int32)
    state[1, :4] = 7
    got, want = run_both(logits, state, 499, D, 3, torch.float32, formulas, children)
    assert assert_parity(got, want) == 2


@pytest.mark.parametrize("dtype,V,at", [("bf16", 8192, [0, 1, 2, 3]), ("bf16", 8192, [1024, 2048, 3072, 1025]),
                                        ("bf16", 8199, [8192, 8195, 8198, 8191]), ("f32", 4099, [4098, 4097, 4096, 5]),
                                        ("f32", 3, [2, 0, 1, 1]), ("bf16", 20001, [5, 7000, 14000, 20000])])
def test_where_the_largest_lie(dtype, V, at):
    r = np.random.default_rng(V)
    logits = np.round(r.standard_normal((1, 4, V))).astype(np.float32)
    logits[0, 0, at] = 9.0          # ties: the lower token id first
    logits[0, 1, at] = [12.0, 11.0, 10.0, 9.0]
    logits[0, 2, at] = [9.0, 10.0, 11.0, 12.0]
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float32
    room = torch.full((1, 4, (V + 7) // 8 * 8 + 8), 1e4, dtype=tdt, device="cuda")
    room[..., :V] = torch.from_numpy(logits)
    K = min(4, V)
    formulas = [[(i, j)] for i in range(4) for j in range(K)]
    children = [[] for _ in formulas]
    state = np.full((1, 4), V, dtype=np.int32)
    got = spiffy.spiffy_draft_blocks(room[..., :V], G.to_dev(state), V, spiffy.draft_graph(formulas, children),
                                     len(formulas), K)
    torch.cuda.synchronize()
    want = drafting.draft_blocks(logits, state, V, formulas, children, len(formulas), K)
    assert assert_parity(got, want) == 1
