"""The step planner and the append over many tokens at once, and releases of long lists, against the
pool oracle bit for bit (tables, reference counts, free pages, lengths): token counts at the edges of
a page, forks in the middle of a page before them (copy on write), vacant slots, a bitmap scanned in
several passes, slots of different lengths; and the rows themselves, read back by a decode step."""
import dataclasses

import numpy as np
import pytest

from oracle.trajectory import OracleRun
from tests.parity import assert_close, assert_pool_equal
from workload.configs import TINY

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("beams,P,prompt,counts", [
    (40, 16, 21, [1, 15, 16, 35, 130]),
    (33, 64, 64, [63, 1, 64, 131]),
    (5, 32, 1, [31, 200, 64, 2]),
    (200, 16, 300, [199, 1, 48]),
])
def test_append_many_tokens(cuda, beams, P, prompt, counts):
    import torch
    from workload.driver import GpuRun
    wl = dataclasses.replace(TINY, beams=beams, page_size=P, prompt_len=prompt, context=prompt + sum(counts) + 8,
                             K=beams // 2)
    g, o = GpuRun(wl), OracleRun(wl, literal_kv=False)
    g.seed()
    o.seed()
    rng = np.random.default_rng(beams)
    for i, n in enumerate(counts):
        g.append(n)
        o.append(n)
        assert_pool_equal(g.pool.read_state(), o.pool, P, means="exact")
        sc = rng.uniform(size=beams).astype(np.float32)
        g.pool.push_scores(torch.from_numpy(sc).cuda())
        o.push_scores(sc)
        g.prune()
        o.prune()
        if i == 1:                           # a list longer than a block, with repeats: only the first counts
            slots = [0, beams - 1] + [beams // 2] * 1100
            g.pool.release(torch.tensor(slots, dtype=torch.int32, device="cuda"))
            o.pool.release(slots)
            assert g.pool.status() == o.pool.status != 0
            g.pool.clear_status()
            o.pool.status = 0
        assert_pool_equal(g.pool.read_state(), o.pool, P, means="exact")
    out = g.decode_step().cpu().numpy()
    ref = o.decode_step()
    for (layer, b) in list(ref)[:: max(1, len(ref) // 12)]:
        assert_close(out[layer, b], ref[(layer, b)], "f32", f"slot {b}")
    assert g.pool.status() == 0


@pytest.mark.parametrize("dtype,P,C", [("f32", 16, 9), ("bf16", 32, 40)])
def test_unequal_lengths(cuda, dtype, P, C):
    """Active slots of different lengths, which only forks from a released parent make (their children
    start empty): the planner's token-by-token form, with copies on write in the same step."""
    import torch
    from oracle.pool import PoolOracle
    from paper_2608_08020_gb300 import binding as B
    from paper_2608_08020_gb300.pool import BeamPool, TORCH_DT
    Hkv, G, D, dt, prompt, width = 2, 2, 64 if dtype == "f32" else 128, TORCH_DT[dtype], 21, 12
    g = torch.Generator(device="cuda").manual_seed(P)
    rnd = lambda *s: torch.randn(s, generator=g, device="cuda").to(dt)
    pool = BeamPool(num_layers=1, num_q_heads=Hkv * G, num_kv_heads=Hkv, head_dim=D, page_size=P, kv_dtype=dtype,
                    num_pages=C * width, max_beams=C, max_pages_per_beam=width)
    ref = PoolOracle(C * width, C, width, P)
    kp, vp = rnd(1, prompt, Hkv, D), rnd(1, prompt, Hkv, D)
    pool.seed(C, prompt, kp, vp)
    ref.seed(C, prompt)
    kv = [[kp[0], vp[0]] for _ in range(C)]              # each slot's rows

    def append(n):
        k, v = rnd(n, C, Hkv, D), rnd(n, C, Hkv, D)
        pool.append_kv(0, n, k, v)
        for _ in range(n):
            assert ref.begin_step()
        for b in range(C):
            if ref.active[b]:
                kv[b] = [torch.cat([x, y[:, b]]) for x, y in zip(kv[b], (k, v))]

    def fork(children):
        parent = np.where(ref.active, np.arange(C), -1).astype(np.int32)
        for s, p in children.items():
            parent[s] = p
            kv[s] = kv[p] if ref.active[p] else [x[:0] for x in kv[p]]
        B.gb_fork_slots(pool.handle, torch.from_numpy(parent).cuda())
        ref.fork_slots(parent)

    append(3)
    gone = [2, 5]
    pool.release(torch.tensor(gone, dtype=torch.int32, device="cuda"))
    ref.release(gone)
    for n, children in ((1, {7: 2, 5: 0}), (15, {8: 7, 3: 6}), (2, {1: 7}), (40, {0: 8, 4: 3, 6: 2})):
        fork(children)
        assert len(set(ref.seq_len[ref.active])) > 1
        append(n)
        assert_pool_equal(pool.read_state(), ref, P)
    q, k, v = rnd(C, Hkv * G, D), rnd(C, Hkv, D), rnd(C, Hkv, D)
    out = torch.full((C, Hkv * G, D), 7.0, device="cuda")
    pool.decode_attention(0, q, k, v, 0.1, out)
    assert ref.begin_step()
    assert_pool_equal(pool.read_state(), ref, P)
    for b in range(C):
        if not ref.active[b]:
            assert not bool(out[b].any())
            continue
        K, V = (torch.cat([x, y[b][None]]).double().repeat_interleave(G, dim=1) for x, y in zip(kv[b], (k, v)))
        p = torch.softmax(torch.einsum("hd,thd->ht", q[b].double(), K) * 0.1, -1)
        assert_close(out[b].cpu().numpy(), torch.einsum("ht,thd->hd", p, V).cpu().numpy(), dtype, f"slot {b}")
    assert pool.status() == 0
