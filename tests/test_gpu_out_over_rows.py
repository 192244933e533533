"""gb_decode_attention whose output lies over its own new K/V rows (one scratch buffer for both): the same
outputs, bit for bit, and the same rows in the pool as with buffers of their own, on every path."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,G,Hkv,C,prompt,flags", [
    ("bf16", 4, 8, 200, 40, 0), ("bf16", 4, 8, 200, 40, 2), ("bf16", 2, 8, 300, 1500, 1), ("f32", 2, 8, 200, 40, 0),
    ("f32", 2, 8, 160, 300, 0), ("bf16", 2, 48, 1024, 20, 0),     # more new rows than the scorer's scratch holds
])
def test_output_over_new_rows(cuda, dtype, G, Hkv, C, prompt, flags):
    import torch
    from paper_2608_08020_gb300.pool import BeamPool, TORCH_DT
    D, layers, dt = 128 if dtype == "bf16" else 64, 2, TORCH_DT[dtype]
    g = torch.Generator(device="cuda").manual_seed(C)
    rnd = lambda *s: torch.randn(s, generator=g, device="cuda").to(dt)
    kp, vp = rnd(layers, prompt, Hkv, D), rnd(layers, prompt, Hkv, D)
    pools = []
    for _ in (0, 1):
        p = BeamPool(num_layers=layers, num_q_heads=Hkv * G, num_kv_heads=Hkv, head_dim=D, page_size=16, kv_dtype=dtype,
                     num_pages=C * 2 + prompt // 16 + 2, max_beams=C, max_pages_per_beam=prompt // 16 + 2)
        p.seed(C, prompt, kp, vp)
        pools.append(p)
    n_out, n_row = C * Hkv * G * D, C * Hkv * D
    buf = torch.empty(n_out, dtype=torch.float32, device="cuda")
    over = buf.view(dt)
    for step in range(3):
        for l in range(layers):
            q, k, v = rnd(C, Hkv * G, D), rnd(C, Hkv, D), rnd(C, Hkv, D)
            want = torch.empty(C, Hkv * G, D, device="cuda")
            pools[0].decode_attention(l, q, k, v, 0.1, want, flags)
            first = 0 if step % 2 else min(n_row // 2, over.numel() - 2 * n_row)
            at = (first, over.numel() - n_row if step % 2 else first + n_row)
            kk, vv = over[at[0]:at[0] + n_row], over[at[1]:at[1] + n_row]
            kk.copy_(k.flatten())
            vv.copy_(v.flatten())
            pools[1].decode_attention(l, q, kk, vv, 0.1, buf, flags)
            assert torch.equal(buf.view_as(want), want), (step, l)
    assert pools[0].status() == pools[1].status() == 0
