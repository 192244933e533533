"""Tournament rounds whose CTAs start at different times: caller-owned rows decode on another stream
meanwhile, on every SM, so a round's CTAs get theirs one by one as those calls' CTAs leave.  Every CTA
must rank the state before the round, whatever the others have written by then (and the caller's mask,
where the pruned flags overwrite it): tables, reference counts, parents and means bit for bit as the
oracle's, for pools with and without segments, at capacity and below it."""
import dataclasses

import numpy as np
import pytest

from tests.parity import assert_pool_equal
from tests.test_gpu_prune import _round, _setup
from tests.test_zz_no_alloc_sizes import _setup as _rows
from workload import gen
from workload.configs import QWEN3_8B_LAYER, TINY

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("base,beams,fanout", [(TINY, 256, 2), (TINY, 100, 4), (QWEN3_8B_LAYER, 512, 3)])
def test_late_ctas_rank_the_same_state(cuda, base, beams, fanout):
    import torch
    wl = dataclasses.replace(base, beams=beams, prompt_len=64, context=1000, K=beams // 2, hidden=256)
    g, o = _setup(wl, grow=60, device_gen=base is not TINY)
    call, _ = _rows("bf16", 4, 8, 32, [2100, 700, 1, 1500] * 8, seed=1)
    side = torch.cuda.Stream()
    for r in range(12):
        if r == 8:                               # vacant slots: the rounds below capacity
            slots = list(range(1, beams, 3))
            g.pool.release(torch.tensor(slots, dtype=torch.int32, device="cuda"))
            o.pool.release(slots)
        scores = gen.uniform([r, 3, beams], beams)
        mask = gen.uniform([r, 4, beams], beams) > 0.3
        g.pruned.copy_(torch.from_numpy(mask.astype(np.uint8)))
        torch.cuda.synchronize()
        with torch.cuda.stream(side):
            for _ in range(8):
                call()
        if r % 4 == 1:                           # the pruned flags over the eligibility mask
            g.pool.push_scores(torch.from_numpy(scores).to(g.dev))
            o.push_scores(scores)
            parent, pruned, _ = (t.cpu().numpy() for t in g.prune(beams // 2, fanout, 0, g.pruned))
            _, parent_o, pruned_o = o.prune(beams // 2, fanout, 0, mask)
            assert np.array_equal(parent, parent_o) and np.array_equal(pruned, pruned_o)
            assert_pool_equal(g.pool.read_state(), o.pool, wl.page_size, means="exact")
        else:
            _round(g, o, scores, K=beams // 2, fanout=fanout)
        torch.cuda.synchronize()
        g.append(3)
        o.append(3)
    assert g.pool.status() == 0
