"""MLP scorer widths at the edges of its 16-byte forms: rows of partials that are and are not
whole 16-byte pieces, one column, one past a tile, one past a pass of a score CTA's threads, and
more k-blocks than the ring has stages."""
import numpy as np
import pytest

from oracle.probe import mlp_probe_score
from tests.parity import assert_close
from tests.test_gpu_mlp import _bf16

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,H,dh", [(3, 64, 1), (129, 1024, 129), (130, 192, 4), (7, 4096, 513), (64, 4096, 516),
                                    (600, 8192, 130)])
def test_mlp_widths_match_oracle(cuda, C, H, dh):
    import torch
    from paper_2608_08020_gb300.pool import BeamPool
    rng = np.random.default_rng(C + H + dh)
    pool = BeamPool(num_layers=1, num_q_heads=4, num_kv_heads=1, head_dim=128, page_size=16, kv_dtype="bf16",
                    num_pages=C * 2 + 8, max_beams=C, max_pages_per_beam=2)
    kp = torch.zeros((1, 16, 1, 128), dtype=torch.bfloat16, device="cuda")
    pool.seed(C, 16, kp, kp)
    h = _bf16(rng.standard_normal((C, H)).astype(np.float32))
    w1 = _bf16((rng.standard_normal((dh, H)) / np.sqrt(H)).astype(np.float32))
    b1 = (rng.standard_normal(dh) * 0.1).astype(np.float32)
    w2 = (rng.standard_normal(dh) / np.sqrt(dh)).astype(np.float32)
    td = lambda a, dt: torch.from_numpy(np.ascontiguousarray(a)).to(dt).cuda()
    score = torch.zeros(C, dtype=torch.float32, device="cuda")
    pool.score_mlp(td(h, torch.bfloat16), td(w1, torch.bfloat16), td(b1, torch.float32), td(w2, torch.float32), 0.1,
                   score_out=score)
    assert_close(score.cpu().numpy(), mlp_probe_score(h, w1, b1, w2, 0.1), "bf16", f"mlp C={C} H={H} d_h={dh}")
    assert pool.status() == 0
