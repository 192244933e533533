"""Large steps of fp32 pools by the records of a pair: one warp merges a few (up to 32, 16 and 8 with G = 2, 4
and 8), the whole CTA more, and a warp's share may end one such pair and begin the next; against fp64, whatever
the values (fp32 sums: 1e-5 of the output's scale)."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,G,Hkv,prompt", [
    (1, 2, 1, 510), (1, 2, 1, 526), (1, 4, 1, 400), (1, 8, 1, 400), (1, 8, 1, 4000),   # a record per chunk
    (3, 4, 2, 3000), (20, 8, 2, 2000), (20, 4, 2, 2005), (50, 2, 8, 333), (153, 8, 8, 250),
])
def test_records_of_a_pair(cuda, C, G, Hkv, prompt):
    import torch
    from paper_2608_08020_gb300.pool import BeamPool
    D, scale = 64, 0.125
    g = torch.Generator(device="cuda").manual_seed(prompt + G)
    rnd = lambda *s: torch.randn(s, generator=g, device="cuda")
    pool = BeamPool(num_layers=2, num_q_heads=Hkv * G, num_kv_heads=Hkv, head_dim=D, page_size=16, kv_dtype="f32",
                    num_pages=C * 2 + prompt // 16 + 2, max_beams=C, max_pages_per_beam=prompt // 16 + 2)
    kp, vp = rnd(2, prompt, Hkv, D), rnd(2, prompt, Hkv, D)
    pool.seed(C, prompt, kp, vp)
    K, V = ([x[l].expand(C, -1, -1, -1) for l in (0, 1)] for x in (kp, vp))
    for step in range(4):
        for l in (0, 1):                        # both counter sets
            q, k, v = 3 * rnd(C, Hkv * G, D), rnd(C, Hkv, D), rnd(C, Hkv, D)
            out = torch.full((C, Hkv * G, D), 7.0, device="cuda")
            pool.decode_attention(l, q, k, v, scale, out)
            K[l], V[l] = torch.cat([K[l], k[:, None]], 1), torch.cat([V[l], v[:, None]], 1)
            kk, vv = (x.double().repeat_interleave(G, dim=2) for x in (K[l], V[l]))
            p = torch.softmax(torch.einsum("chd,cthd->cht", q.double(), kk) * scale, -1)
            ref = torch.einsum("cht,cthd->chd", p, vv)
            assert bool(((out.double() - ref).abs() <= 1e-5 * (1 + ref.abs())).all()), (step, l)
            assert int(pool.meta[4 * 14:4 * 15].view(torch.int32)) == 0     # the even split
    assert pool.status() == 0


def test_shares_across_vacant_slots(cuda):
    """A warp's share that ends one active slot's chunks and begins the next one's, a hundred vacant slots on."""
    import torch
    from paper_2608_08020_gb300.pool import BeamPool
    slots, G, Hkv, D, prompt, keep = 1024, 2, 8, 64, 1000, list(range(7, 1024, 100))
    g = torch.Generator(device="cuda").manual_seed(1)
    rnd = lambda *s: torch.randn(s, generator=g, device="cuda")
    pool = BeamPool(num_layers=1, num_q_heads=Hkv * G, num_kv_heads=Hkv, head_dim=D, page_size=16, kv_dtype="f32",
                    num_pages=80 + slots, max_beams=slots, max_pages_per_beam=64)
    kp, vp = rnd(1, prompt, Hkv, D), rnd(1, prompt, Hkv, D)
    pool.seed(slots, prompt, kp, vp)
    gone = torch.ones(slots, dtype=torch.bool, device="cuda")
    gone[keep] = False
    pool.release(torch.nonzero(gone).flatten().int())
    q, k, v = rnd(slots, Hkv * G, D), rnd(slots, Hkv, D), rnd(slots, Hkv, D)
    out = torch.full((slots, Hkv * G, D), 7.0, device="cuda")
    pool.decode_attention(0, q, k, v, 0.125, out)
    assert int(pool.meta[4 * 14:4 * 15].view(torch.int32)) == 0 and not bool(out[gone].any())
    K, V = (torch.cat([x[0].expand(len(keep), -1, -1, -1), y[keep][:, None]], 1).double().repeat_interleave(G, dim=2)
            for x, y in ((kp, k), (vp, v)))
    p = torch.softmax(torch.einsum("chd,cthd->cht", q[keep].double(), K) * 0.125, -1)
    ref = torch.einsum("cht,cthd->chd", p, V)
    assert bool(((out[keep].double() - ref).abs() <= 1e-5 * (1 + ref.abs())).all())
    assert pool.status() == 0
