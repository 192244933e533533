"""Small steps (the form that merges inside single CTAs) against fp64: their probabilities enter P.V as
two bf16 terms, so an output is off by at most 2^-17 sum p |v| and what fp32 scores and sums add (about
2e-6 of an output row's 2-norm measured): 2e-5 of the 2-norm allowed, where one rounding to bf16 gives 1e-3.
G = 2, 4 and 8 heads per KV head, teams of one and of several warps, one chunk and several."""
import math

import pytest

pytestmark = pytest.mark.gpu
CTL_TEAM, CTL_TEAM_PER_BEAM = 14, 15         # control words of the metadata buffer (internal.cuh)


@pytest.mark.parametrize("flags", ["auto", "per_beam"])
@pytest.mark.parametrize("C,G,Hkv,P,prompt", [(3, 2, 1, 16, 5), (9, 4, 2, 64, 130), (40, 8, 4, 32, 310),
                                              (300, 4, 8, 16, 60), (7, 2, 2, 16, 900), (5, 8, 1, 16, 15)])
def test_probabilities_keep_sixteen_bits(cuda, C, G, Hkv, P, prompt, flags):
    import torch
    from paper_2608_08020_gb300 import binding as B
    from paper_2608_08020_gb300.pool import BeamPool
    D, T, scale = 128, prompt + 3, 1 / math.sqrt(128)
    g = torch.Generator(device="cuda").manual_seed(C + G)
    rnd = lambda *s: torch.randn(s, generator=g, device="cuda").to(torch.bfloat16)
    pool = BeamPool(num_layers=1, num_q_heads=Hkv * G, num_kv_heads=Hkv, head_dim=D, page_size=P, kv_dtype="bf16",
                    num_pages=C * 2 + T // P + 4 + C, max_beams=C, max_pages_per_beam=T // P + 2)
    kp, vp = rnd(1, prompt, Hkv, D), rnd(1, prompt, Hkv, D)
    pool.seed(C, prompt, kp, vp)
    K, V = (x[0].expand(C, -1, -1, -1) for x in (kp, vp))
    for _ in range(3):
        q, k, v = 2 * rnd(C, Hkv * G, D), rnd(C, Hkv, D), rnd(C, Hkv, D)
        out = torch.full((C, Hkv * G, D), 7.0, device="cuda")
        pool.decode_attention(0, q, k, v, scale, out, B.GB_PATH_AUTO if flags == "auto" else B.GB_PATH_PER_BEAM)
        K, V = torch.cat([K, k[:, None]], 1), torch.cat([V, v[:, None]], 1)
        kk, vv = (x.double().repeat_interleave(G, dim=2) for x in (K, V))
        p = torch.softmax(torch.einsum("chd,cthd->cht", q.double(), kk) * scale, -1)
        ref = torch.einsum("cht,cthd->chd", p, vv)
        err = (out.double() - ref).norm(dim=-1) / ref.norm(dim=-1)
        assert float(err.max()) <= 2e-5, float(err.max())
        ctl = pool.meta[:128].view(torch.int32).tolist()
        assert ctl[CTL_TEAM if flags == "auto" else CTL_TEAM_PER_BEAM] > 0     # the small-step form was taken
    assert pool.status() == 0
