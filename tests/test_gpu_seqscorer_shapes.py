"""The sequence scorer's products on both sides of d_model 512: fused ones at the edges of their tiles
(row tiles of 32, 64 and 128 slots with a ragged last one, K of several passes with a partial last
one, one column tile per head half) and K-split ones with their epilogues; against the oracle over forks and releases, as the search test does."""
import pytest

from tests.test_gpu_seqscorer import test_scorer_matches_oracle_over_forks_and_releases as over_a_search

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,H,F,L,Hq,Hkv,steps,P", [
    (33, 128, 64, 1, 2, 1, 4, 16),         # d_model 256, the narrowest FFN
    (300, 256, 1472, 1, 4, 1, 3, 16),      # d_model 512: 64- and 128-row tiles, a partial pass of K
    (513, 128, 2048, 1, 2, 1, 2, 16),      # rows past the last tile, two passes of K at 32-row tiles
    (300, 256, 1472, 1, 8, 2, 3, 16),      # d_model 1024: K-split products
    (70, 192, 640, 2, 16, 4, 3, 32),       # d_model 2048
])
def test_products_match_oracle(cuda, C, H, F, L, Hq, Hkv, steps, P):
    over_a_search(cuda, C, H, F, L, Hq, Hkv, steps, P)
