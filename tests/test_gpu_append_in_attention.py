"""Decode steps that append inside the attention launch, mixed with layers appended alone.

A step's layers are decoded on the three paths or appended with gb_append_kv, in every mix, with forks
in the middle of a page, so that steps after them copy the shared tail page on write.  Short contexts
take the form that merges inside single CTAs, except on GB_PATH_GROUPED; long ones take the roles and
the even splits, which use the attention launches' two counter sets, so the sets are used in every
order, with launches that leave them alone and appended layers between.  Each decoded layer is compared
with fp64 attention over the K/V each beam holds, and at the end the per-beam path re-reads everything
the steps wrote.

Tolerances: fp32 pools 1e-5 (fp32 sums); bf16 pools 2e-3 + 1e-2 |ref| (probabilities rounded to
8 bits), the bounds of the other decode tests.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,G,P,layers,prompt", [
    ("bf16", 4, 16, 3, 21), ("bf16", 2, 64, 2, 64), ("bf16", 8, 32, 1, 47), ("bf16", 4, 64, 3, 111),
    ("f32", 2, 16, 2, 21), ("f32", 4, 64, 1, 63),
    ("bf16", 4, 16, 3, 2700), ("bf16", 2, 64, 2, 2690), ("bf16", 8, 32, 1, 2715), ("f32", 2, 16, 3, 1500), ("f32", 8, 32, 2, 1510),
])
def test_mixed_steps(cuda, dtype, G, P, layers, prompt):
    import torch
    from paper_2608_08020_gb300 import binding as B
    from paper_2608_08020_gb300.pool import BeamPool, TORCH_DT
    C, Hkv, D = 7, 2, 128 if dtype == "bf16" else 64
    Hq, dt, scale = Hkv * G, TORCH_DT[dtype], 0.125
    g = torch.Generator(device="cuda").manual_seed(P * 31 + G + layers)
    rnd = lambda *s: torch.randn(s, generator=g, device="cuda").to(dt)
    T, long = prompt + 60, prompt > 1000
    forms = set()
    pool = BeamPool(num_layers=layers, num_q_heads=Hq, num_kv_heads=Hkv, head_dim=D, page_size=P, kv_dtype=dtype,
                    num_pages=C * (T // P + 3), max_beams=C, max_pages_per_beam=T // P + 2)
    K, V = (torch.zeros(layers, C, T, Hkv, D, dtype=dt, device="cuda") for _ in (0, 1))
    kp, vp = rnd(layers, prompt, Hkv, D), rnd(layers, prompt, Hkv, D)
    K[:, :, :prompt], V[:, :, :prompt] = kp[:, None], vp[:, None]
    pool.seed(C, prompt, kp, vp)
    at = prompt

    def decode(layer, flags):
        q, k, v = rnd(C, Hq, D), rnd(C, Hkv, D), rnd(C, Hkv, D)
        out = torch.full((C, Hq, D), 7.0, device="cuda")
        pool.decode_attention(layer, q, k, v, scale, out, flags)
        K[layer, :, at], V[layer, :, at] = k, v
        kk, vv = (x[layer, :, :at + 1].double().repeat_interleave(G, dim=2) for x in (K, V))
        s = torch.einsum("chd,cthd->cht", q.double(), kk) * scale
        ref = torch.einsum("cht,cthd->chd", torch.softmax(s, -1), vv)
        err = (out.double() - ref).abs()
        tol = 1e-5 if dtype == "f32" else 2e-3 + 1e-2 * ref.abs()
        assert bool((err <= tol).all()), (layer, at, float(err.max()))
        ctl = pool.meta[:128].view(torch.int32).tolist()
        team = ctl[15] if flags == B.GB_PATH_PER_BEAM and dtype == "bf16" else ctl[14]  # internal.cuh
        if dtype == "f32" or flags == B.GB_PATH_PER_BEAM or (flags == B.GB_PATH_AUTO and not long):
            forms.add(team > 0)     # GB_PATH_GROUPED takes the roles whatever the size

    rng = np.random.default_rng(3)
    for step in range(36):
        if step in (5, 6, 17, 18, 30):       # forks; 5/6 and 17/18: two rounds with one step between
            parent = np.arange(C, dtype=np.int32)
            child = rng.choice(C, 3, replace=False)
            rest = np.setdiff1d(np.arange(C), child)
            parent[child] = rng.choice(rest, 3)
            B.gb_fork_slots(pool.handle, torch.from_numpy(parent).cuda())
            for X in (K, V):
                X[:, child] = X[:, parent[child]]
        kind = step % 4
        n = 3 if kind == 3 and step % 8 == 3 else 1
        for layer in range(layers):
            alone = n > 1 or (kind == 1 and layer % 2 == 0) or (kind == 2 and layer == layers - 1)
            if alone:
                k, v = rnd(n, C, Hkv, D), rnd(n, C, Hkv, D)
                pool.append_kv(layer, n, k, v)
                K[layer, :, at:at + n], V[layer, :, at:at + n] = k.transpose(0, 1), v.transpose(0, 1)
            else:
                decode(layer, (B.GB_PATH_AUTO, B.GB_PATH_GROUPED, B.GB_PATH_AUTO, B.GB_PATH_GROUPED,
                               B.GB_PATH_PER_BEAM)[step % 5])
        at += n
    for layer in range(layers):
        decode(layer, B.GB_PATH_PER_BEAM)
    assert forms == {not long}
    assert pool.status() == 0
