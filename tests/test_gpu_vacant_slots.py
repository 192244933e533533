"""Pools with many vacant slots.  An fp32 pool decodes as one of just the active ones does: the same split of
the work (the control word of the step's team form), and the same values, against fp64 (fp32 sums: 1e-5).
A bf16 pool's small steps skip the vacant ones of a team's next 32 pairs at once: active slots anywhere
among up to 1024, runs of vacant ones of more than 32 pairs too, whatever the team (two bf16 terms of P:
2e-5 of a row's 2-norm), zeros for the vacant ones."""
import math

import pytest

pytestmark = pytest.mark.gpu
CTL_TEAM = 14        # control word of the metadata buffer (internal.cuh)


@pytest.mark.parametrize("beams,G,Hkv,prompt", [(8, 2, 2, 260), (4, 4, 1, 1000), (16, 2, 8, 1500), (8, 8, 2, 70),
                                                (3, 2, 4, 3000)])
def test_vacant_slots_do_not_change_the_split(cuda, beams, G, Hkv, prompt):
    import torch
    from paper_2608_08020_gb300.pool import BeamPool
    D, P, scale, teams, outs = 64, 16, 1 / math.sqrt(64), [], []
    for slots in (beams, 512, 1024):
        g = torch.Generator(device="cuda").manual_seed(beams + prompt)
        rnd = lambda *s: torch.randn(s, generator=g, device="cuda")
        kp, vp = rnd(1, prompt, Hkv, D), rnd(1, prompt, Hkv, D)
        q, k, v = (rnd(beams, n * Hkv, D) for n in (G, 1, 1))
        q, k, v = (torch.cat([x, torch.full((slots - beams, *x.shape[1:]), float("nan"), device="cuda")]) for x in (q, k, v))
        pool = BeamPool(num_layers=1, num_q_heads=Hkv * G, num_kv_heads=Hkv, head_dim=D, page_size=P, kv_dtype="f32",
                        num_pages=prompt // P + 2 + beams, max_beams=slots, max_pages_per_beam=prompt // P + 2)
        pool.seed(beams, prompt, kp, vp)
        out = torch.full((slots, Hkv * G, D), 7.0, device="cuda")
        pool.decode_attention(0, q, k, v, scale, out)
        assert pool.status() == 0 and not bool(out[beams:].any())
        teams.append(int(pool.meta[4 * CTL_TEAM:4 * CTL_TEAM + 4].view(torch.int32)))
        outs.append(out[:beams])
        K, V = (torch.cat([x[0].expand(beams, -1, -1, -1), y[:beams, None]], 1).double().repeat_interleave(G, dim=2)
                for x, y in ((kp, k), (vp, v)))
        p = torch.softmax(torch.einsum("chd,cthd->cht", q[:beams].double(), K) * scale, -1)
        err = (out[:beams].double() - torch.einsum("cht,cthd->chd", p, V)).abs().max()
        assert float(err) <= 1e-5, (slots, float(err))
    assert teams[1:] == teams[:1] * 2, teams
    assert torch.equal(outs[0], outs[1]) and torch.equal(outs[0], outs[2])


@pytest.mark.parametrize("flags", ["auto", "per_beam"])
@pytest.mark.parametrize("slots,G,Hkv,keep", [
    (1024, 4, 8, [3, 500, 901, 1000, 1023]),     # teams of 12 warps, runs of up to 32 of their pairs
    (1024, 2, 8, list(range(5, 1024, 19))),      # all on the same CTAs
    (700, 8, 4, list(range(0, 700, 2))),         # every other slot, smaller teams
    (1024, 2, 16, [1022]),                       # runs of more than 32, one slot near the end
])
def test_active_slots_anywhere(cuda, slots, G, Hkv, keep, flags):
    import torch
    from paper_2608_08020_gb300 import binding as B
    from paper_2608_08020_gb300.pool import BeamPool
    D, P, prompt, scale = 128, 16, 100, 1 / math.sqrt(128)
    g = torch.Generator(device="cuda").manual_seed(slots + G)
    rnd = lambda *s: torch.randn(s, generator=g, device="cuda").to(torch.bfloat16)
    pool = BeamPool(num_layers=2, num_q_heads=Hkv * G, num_kv_heads=Hkv, head_dim=D, page_size=P, kv_dtype="bf16",
                    num_pages=prompt // P + 2 + slots, max_beams=slots, max_pages_per_beam=prompt // P + 2)
    kp, vp = rnd(2, prompt, Hkv, D), rnd(2, prompt, Hkv, D)
    pool.seed(slots, prompt, kp, vp)
    gone = torch.ones(slots, dtype=torch.bool)
    gone[keep] = False
    pool.release(torch.nonzero(gone).flatten().int().cuda())
    for l in (0, 1):
        q, k, v = rnd(slots, Hkv * G, D), rnd(slots, Hkv, D), rnd(slots, Hkv, D)
        for x in (q, k, v):
            x[gone.cuda()] = float("nan")
        out = torch.full((slots, Hkv * G, D), 7.0, device="cuda")
        pool.decode_attention(l, q, k, v, scale, out, B.GB_PATH_AUTO if flags == "auto" else B.GB_PATH_PER_BEAM)
        assert int(pool.meta[4 * (14 if flags == "auto" else 15):][:4].view(torch.int32)) > 0
        assert not bool(out[gone.cuda()].any())
        K, V = (torch.cat([x[l].expand(len(keep), -1, -1, -1), y[keep][:, None]], 1).double().repeat_interleave(G, dim=2)
                for x, y in ((kp, k), (vp, v)))
        p = torch.softmax(torch.einsum("chd,cthd->cht", q[keep].double(), K) * scale, -1)
        ref = torch.einsum("cht,cthd->chd", p, V)
        err = (out[keep].double() - ref).norm(dim=-1) / ref.norm(dim=-1)
        assert float(err.max()) <= 2e-5, float(err.max())
    assert pool.status() == 0
