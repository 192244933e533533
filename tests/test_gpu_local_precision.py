"""Small steps (the form that merges inside single CTAs) against fp64: their probabilities enter P.V as
two bf16 terms, so an output is off by at most 2^-16 sum p |v| and what fp32 scores and sums add (a few
1e-6 of an output row's 2-norm measured): 2e-5 of the 2-norm allowed, where one rounding to bf16 gives 1e-3.
G = 2, 4 and 8 heads per KV head, teams of one and of several warps, one chunk and several.  Infinities
and NaN in V come out as the sum of p V has them, for probabilities that are exact in bf16 too."""
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


@pytest.mark.parametrize("G,Hkv,flags", [(2, 2, 0), (4, 2, 1), (8, 1, 0), (8, 2, 1)])
def test_infinite_values(cuda, G, Hkv, flags):
    import torch
    from paper_2608_08020_gb300.pool import BeamPool
    C, D, P, prompt, scale = 6, 128, 16, 70, 1 / math.sqrt(128)
    g = torch.Generator(device="cuda").manual_seed(G)
    rnd = lambda *s: torch.randn(s, generator=g, device="cuda").to(torch.bfloat16)
    pool = BeamPool(num_layers=1, num_q_heads=Hkv * G, num_kv_heads=Hkv, head_dim=D, page_size=P, kv_dtype="bf16",
                    num_pages=64, max_beams=C, max_pages_per_beam=prompt // P + 2)
    kp, vp = rnd(1, prompt, Hkv, D), rnd(1, prompt, Hkv, D)
    for t in range(prompt):                      # +inf, -inf and both (NaN) in dims of their own, in every chunk
        vp[0, t, :, t % 40] = math.inf
        vp[0, t, :, 40 + t % 40] = -math.inf
    vp[0, 3, :, 80] = math.inf
    vp[0, 60, :, 80] = -math.inf
    vp[0, 33, :, 81] = math.nan
    pool.seed(C, prompt, kp, vp)
    q, k, v = 2 * rnd(C, Hkv * G, D), rnd(C, Hkv, D), rnd(C, Hkv, D)
    q[:2] = 0                                    # every probability the same, exact in bf16
    out = torch.full((C, Hkv * G, D), 7.0, device="cuda")
    pool.decode_attention(0, q, k, v, scale, out, flags)
    K, V = (torch.cat([x[0].expand(C, -1, -1, -1), y[:, None]], 1).double().repeat_interleave(G, dim=2) for x, y in ((kp, k), (vp, v)))
    p = torch.softmax(torch.einsum("chd,cthd->cht", q.double(), K) * scale, -1)
    ref = (p.transpose(1, 2)[..., None] * V).sum(1)
    assert bool(torch.isinf(ref).any()) and bool(torch.isnan(ref).any())
    for f in (torch.isnan, torch.isposinf, torch.isneginf):
        assert torch.equal(f(out), f(ref)), f.__name__
    ok = torch.isfinite(ref)
    assert float((out.double() - ref)[ok].norm() / ref[ok].norm()) <= 2e-5
    assert pool.status() == 0 and int(pool.meta[4 * (14 + flags):][:4].view(torch.int32)) > 0
