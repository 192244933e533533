"""The sequence scorer at its size limits: hidden_dim and d_model of 12288 run, the next sizes are refused as
unsupported.  The largest d_model against the definition, with the transformer's output products zero (the
stream stays GELU(W_in LN(h)); the score bound is the scorer test's)."""
import numpy as np
import pytest

from oracle.seqscorer import gelu, layer_norm
from tests.test_gpu_seqscorer import ATOL
from tests.test_gpu_seqscorer import test_scorer_matches_oracle_over_forks_and_releases as over_a_search
from workload.scorer_weights import _bf16

pytestmark = pytest.mark.gpu


def test_largest_hidden_dim(cuda):
    over_a_search(cuda, 8, 12288, 128, 1, 2, 1, 4, 16)


def test_largest_d_model(cuda):
    import torch
    from paper_2608_08020_gb300.seqscorer import SeqScorer
    C, H, F, Hq, Hkv, d = 5, 64, 64, 96, 12, 12288
    rng = np.random.default_rng(1)
    ln = lambda n: ((1 + 0.1 * rng.standard_normal(n)).astype(np.float32), (0.1 * rng.standard_normal(n)).astype(np.float32))
    zero = lambda r, c: np.broadcast_to(np.float32(0), (r, c))
    w = {"ln_in": ln(H), "w_in": _bf16(rng.standard_normal((d, H)) / np.sqrt(H)), "layers": [
            {"ln1": ln(d), "wq": zero(d, d), "wk": zero(Hkv * 128, d), "wv": zero(Hkv * 128, d), "wo": zero(d, d),
             "ln2": ln(d), "w1": zero(F, d), "w3": zero(F, d), "w2": zero(d, F)}],
         "ln_out": ln(d), "w_out": (rng.standard_normal(d) / np.sqrt(d)).astype(np.float32), "b_out": 0.1,
         "n_q_heads": Hq, "n_kv_heads": Hkv}
    sc = SeqScorer(w, hidden_dim=H, ffn_dim=F, max_beams=C, max_steps=3)
    sc.seed(torch.from_numpy(rng.standard_normal(H).astype(np.float32)).to(torch.bfloat16).cuda(), C - 1)
    score = torch.full((C,), 7.0, device="cuda")
    for _ in range(2):
        h = _bf16(rng.standard_normal((C, H)).astype(np.float32))
        sc.step(torch.from_numpy(h).to(torch.bfloat16).cuda(), score)
        z = layer_norm(gelu(layer_norm(h, *w["ln_in"]) @ w["w_in"].astype(np.float64).T), *w["ln_out"])
        want = 1 / (1 + np.exp(-(z @ w["w_out"].astype(np.float64) + w["b_out"])))
        got = score.cpu().numpy()
        assert np.abs(got[:-1] - want[:-1]).max() <= ATOL and got[-1] == 0
    assert sc.pool.status() == 0


@pytest.mark.parametrize("H,Hq,Hkv", [(12352, 2, 1), (64, 98, 49)])
def test_larger_sizes_are_refused(cuda, H, Hq, Hkv):
    import torch
    from paper_2608_08020_gb300 import binding as B
    from paper_2608_08020_gb300.pool import BeamPool
    pool = BeamPool(num_layers=1, num_q_heads=Hq, num_kv_heads=Hkv, head_dim=128, page_size=16, kv_dtype="bf16",
                    num_pages=16, max_beams=4, max_pages_per_beam=4)
    buf = torch.zeros(1024, dtype=torch.uint8, device="cuda")
    with pytest.raises(B.GambitError) as e:
        B.gb_scorer_seed(pool.handle, B.GbScorerConfig(H, 64), buf, buf, buf, 4)
    assert e.value.code == B.GB_ERR_UNSUPPORTED
    assert pool.status() == 0
