"""The sequence scorer's fused products at the edges of their tiles: row tiles of 32, 64 and 128 slots
with a ragged last one, K of several passes with a partial last one (ffn 1472, d_model 2048), one
column tile per head half; against the oracle over forks and releases, as the search test does."""
import pytest

from tests.test_gpu_seqscorer import test_scorer_matches_oracle_over_forks_and_releases as over_a_search

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,H,F,L,Hq,Hkv,steps,P", [
    (33, 128, 64, 1, 2, 1, 4, 16),         # d_model 256, the narrowest FFN
    (300, 256, 1472, 1, 8, 2, 3, 16),      # 64- and 128-row tiles, a partial pass of K
    (70, 192, 640, 2, 16, 4, 3, 32),       # d_model 2048: four passes of the LayerNorm rows
])
def test_fused_products_match_oracle(cuda, C, H, F, L, Hq, Hkv, steps, P):
    over_a_search(cuda, C, H, F, L, Hq, Hkv, steps, P)
