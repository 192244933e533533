"""A large step of an fp32 pool while other kernels hold part of the SMs for longer than the library's
wait limit (2 s): its CTAs run in waves, and none may wait for one that has not got an SM.  160 x 8 pairs,
each a little more than one warp's share, so that a CTA that merged what others wrote would need the
last CTAs' records.  Against fp64 (fp32 sums: 1e-5)."""
import math
import time

import pytest

pytestmark = pytest.mark.gpu


def test_fp32_step_needs_no_residency(cuda):
    import torch
    from paper_2608_08020_gb300.pool import BeamPool
    C, G, Hkv, D, prompt, scale = 160, 2, 8, 64, 300, 0.125
    g = torch.Generator(device="cuda").manual_seed(5)
    rnd = lambda *s: torch.randn(s, generator=g, device="cuda")
    pool = BeamPool(num_layers=1, num_q_heads=Hkv * G, num_kv_heads=Hkv, head_dim=D, page_size=16, kv_dtype="f32",
                    num_pages=C * 2 + 40, max_beams=C, max_pages_per_beam=32)
    kp, vp = rnd(1, prompt, Hkv, D), rnd(1, prompt, Hkv, D)
    pool.seed(C, prompt, kp, vp)
    K, V = (x[0].expand(C, -1, -1, -1) for x in (kp, vp))
    streams = [torch.cuda.Stream(priority=-(i // 32)) for i in range(64)]
    for held in (False, True):
        q, k, v, out = rnd(C, Hkv * G, D), rnd(C, Hkv, D), rnd(C, Hkv, D), torch.zeros(C, Hkv * G, D, device="cuda")
        torch.cuda.synchronize()
        if held:
            for s in streams:                  # a thread on an SM of its own each, 3 s and more at 2.07 GHz
                with torch.cuda.stream(s):
                    torch.cuda._sleep(6_500_000_000)
            time.sleep(0.1)
        t0 = time.perf_counter()
        pool.decode_attention(0, q, k, v, scale, out)
        assert pool.status() == 0
        took = time.perf_counter() - t0
        assert took < 1.5, took
        assert int(pool.meta[4 * 14:4 * 15].view(torch.int32)) == 0     # the even split
        torch.cuda.synchronize()
        K, V = torch.cat([K, k[:, None]], 1), torch.cat([V, v[:, None]], 1)
        kk, vv = (x.double().repeat_interleave(G, dim=2) for x in (K, V))
        p = torch.softmax(torch.einsum("chd,cthd->cht", q.double(), kk) * scale, -1)
        err = (out.double() - torch.einsum("cht,cthd->chd", p, vv)).abs().max()
        assert float(err) <= 1e-5, float(err)
