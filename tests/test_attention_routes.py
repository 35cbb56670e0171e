"""Which of its kernels the tensor-core attention takes (attention_routes.py)."""
import pytest

from paper_2509_18085_b200 import spiffy
import attention_routes as R


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
