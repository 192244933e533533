"""The step planner and the append over many tokens at once, and releases of long lists, against the
pool oracle bit for bit (tables, reference counts, free pages, lengths): token counts at the edges of
a page, forks in the middle of a page before them (copy on write), vacant slots, a bitmap scanned in
several passes; and the rows themselves, read back by a decode step."""
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
