"""Which of its kernels the tensor-core attention takes (attention_routes.py)."""
import pytest

from paper_2509_18085_b200 import spiffy
from paper_2509_18085_b200 import workloads as W
import attention_routes as R
import attention_shapes as shapes
import test_gpu_attention as parity
import test_gpu_attention_d64 as d64
import test_gpu_attention_pair as pair
import test_gpu_attention_splits as splits
import test_gpu_canaries as canaries
import test_gpu_side_by_side as side
import test_gpu_timeouts as timeouts


@pytest.mark.parametrize("B,N,L,P,Hq,Hkv,d,alone,beside", [
    (1, 2, 32, 100, 73, 73, 128, "pair", "pair"), (1, 2, 32, 100, 74, 74, 128, "pair", "one tile"),
    (1, 2, 32, 512, 73, 73, 128, "pair", "pair"), (1, 2, 32, 512, 74, 74, 128, "pair", "one tile"),
    (1, 2, 32, 1200, 74, 74, 128, "pair", "pair"),          # long enough that pairs are sooner done, late or not
    (2, 2, 32, 512, 36, 36, 128, "pair", "pair"), (2, 2, 32, 512, 37, 37, 128, "pair", "one tile"),
    (4, 2, 32, 512, 18, 18, 128, "pair", "pair"), (4, 16, 32, 4096, 32, 32, 128, "two tiles", "two tiles"),
    (5, 4, 16, 512, 29, 29, 128, "one tile", "one tile"),   # 145 of 148, and no better plan
    (1, 2, 32, 512, 73, 73, 64, "pair", "pair"), (1, 2, 32, 512, 74, 74, 64, "pair", "one tile"),
    (1, 8, 32, 100, 73, 73, 128, "one tile", "one tile"), (1, 8, 32, 100, 74, 74, 128, "one tile", "two tiles"),
    (1, 8, 32, 1000, 74, 74, 128, "one tile", "one tile"),
    (1, 146, 32, 512, 2, 2, 128, "pair", "one tile")])
def test_a_decisions_end_beside_the_call_holds_multiprocessors(B, N, L, P, Hq, Hkv, d, alone, beside):
    """One a sequence: a plan that needs them all is one that waits."""
    assert R.route(B, N, L, P, Hq, Hkv, d=d) == alone
    assert R.route(B, N, L, P, Hq, Hkv, d=d, flags=spiffy.ATTN_INDEPENDENT) == beside


@pytest.mark.parametrize("route,shape,d", shapes.SHAPES + shapes.GROWING + shapes.CHAINS)
def test_shapes_take_the_routes_that_they_stand_for(route, shape, d):
    assert R.route(*shape, d=d) == route


@pytest.mark.parametrize("flags", [0, spiffy.ATTN_EARLY_DEPENDENTS])
def test_every_route_has_shapes_at_both_head_dimensions(flags):
    routes = {"pair", "one tile", "two tiles", "cluster of 2", "cluster of 4", "cluster of 8", "two tiles, then pair",
              "two tiles, then one tile"}
    for d in (64, 128):
        assert {R.route(*s, d=d, flags=flags) for _, s, hd in shapes.SHAPES if hd == d} == routes


def claimed(test, names):
    (args,) = [m.args[1] for m in test.pytestmark if m.name == "parametrize" and m.args[0] == names]
    return args


def test_what_the_other_tests_say_of_their_shapes():
    """The routes named in the comments of the parity tests."""
    at = "B,N,L,P,Hq,Hkv"
    got = [R.route(*s) for s in claimed(splits.test_parity, at)]
    assert got == ["pair"] * 6 + ["cluster of 8", "pair", "pair", "pair", "one tile", "two tiles", "two tiles"]
    got = [R.route(*s) for s in claimed(splits.test_last_round_in_a_launch_of_its_own, at)]
    assert got == ["two tiles, then pair", "two tiles, then one tile", "two tiles, then one tile", "two tiles"]
    got = [R.route(*s, d=64) for s in claimed(d64.test_parity, at)]
    assert got == ["pair"] * 6 + ["cluster of 8", "one tile", "two tiles", "pair", "pair", "one tile", "cluster of 8"]
    pairs = claimed(pair.test_parity, at)
    assert (1, 9, 34, 128 * 12 - 3, 28, 4) in pairs
    assert [s for s in pairs if R.route(*s) != "pair"] == [(1, 3, 17, 128 * 12 - 3, 28, 4)]
    assert [s for s in pairs if R.route(*s, d=64) != "pair"] == [(2, 4, 32, 128 * 6, 3, 3), (1, 3, 17, 128 * 12 - 3, 28, 4)]
    for P, N, L in claimed(parity.test_cluster_pairs_with_even_and_odd_tile_counts, "prefix_len,n_nodes,block_len"):
        assert R.route(1, N, L, P, 16, 16) == ("cluster of 4" if P > 2000 else "pair")
    got = []
    for index, n_nodes, over in claimed(timeouts.test_attention_gives_up_when_its_mbarrier_waits_may_not_poll,
                                        "index,n_nodes,over"):
        c = W.config(index, n_nodes, **over)
        got.append(R.route(c.batch, c.n_nodes, c.block_len, c.prefix_len, c.n_q_heads, c.n_kv_heads, d=c.head_dim))
    assert got == ["cluster of 8", "pair", "pair", "one tile", "two tiles, then pair"]
    keys = ("batch", "n_nodes", "block_len", "prefix_len", "n_q_heads", "n_kv_heads", "head_dim")
    got = [R.route(*(s[k] for k in keys[:-1]), d=s["head_dim"]) for s, dtype in canaries.ATTENTION_SHAPES if dtype == "bf16"]
    assert got == ["pair", "pair", "pair", "one tile", "pair", "two tiles", "pair", "two tiles", "cluster of 8"]
    beside = [s for s in claimed(side.test_same_bits_as_one_after_the_other, at + ",d,V,dtype") if s[-1] == "bf16"]
    got = [R.route(*s[:6], d=s[6], flags=spiffy.ATTN_INDEPENDENT) for s in beside]
    assert got == ["pair", "pair", "two tiles, then one tile", "two tiles", "two tiles, then pair", "two tiles, then one tile"]
    assert got == [R.route(*s[:6], d=s[6]) for s in beside]  # else the bits need not be the same
