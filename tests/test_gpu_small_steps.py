"""Small steps on every path against the oracle: the default path takes them inside single CTAs
(local.cuh), GB_PATH_GROUPED sends the same trees through the grouped and per-beam roles.

Beam counts and head counts are at the edges of the team sizes (one pair; fewer pairs than CTAs;
more pairs than warps, so that a warp takes several), contexts from one chunk to beyond a page-id
window of 32 chunks per warp; released slots.

Tolerance: the kernels round each probability to bf16 (relative error at most 2^-9; its sum stays
fp32), so an output is off by at most 2^-9 sum p |v| <= 2^-9 max |v|, with |v| <= 2 sqrt(3) for the
generator's values, and over a whole row (roundings independent, 2^-9 / sqrt(3) each) by about 1.1e-3
of its 2-norm: 4e-3 allowed.  A few elements in a million pass 2e-3 at contexts of some 30 tokens."""
import dataclasses

import numpy as np
import pytest

from oracle.trajectory import OracleRun
from paper_2608_08020_gb300 import binding as B
from tests.parity import assert_pool_equal
from workload.configs import QWEN3_8B_LAYER

pytestmark = pytest.mark.gpu
BOUND = 2.0 ** -9 * 2 * 3 ** 0.5 + 1e-5


def assert_rounded(got, ref, what):
    err = np.abs(np.asarray(got, np.float64) - ref)
    assert float(err.max()) <= BOUND, (what, float(err.max()))
    assert np.linalg.norm(err) <= 4e-3 * np.linalg.norm(ref), (what, np.linalg.norm(err) / np.linalg.norm(ref))


@pytest.mark.parametrize("beams,Hq,Hkv,P,prompt,context,interval", [
    (1, 2, 1, 16, 1, 20, 1 << 30),          # one pair, one chunk, then two
    (2, 8, 1, 64, 6600, 6607, 1 << 30),     # two pairs, long runs: page-id windows beyond 32 chunks
    (8, 4, 2, 16, 72, 210, 40),             # G = 2
    (16, 32, 8, 64, 111, 330, 88),          # 64-token pages, forks in the middle of a page
    (8, 16, 2, 32, 72, 208, 56),            # G = 8
    (300, 32, 8, 16, 33, 90, 24),           # 2400 pairs: more than the GPU's warps
])
@pytest.mark.parametrize("flags", ["auto", "grouped"])
def test_small_steps_match_oracle(cuda, beams, Hq, Hkv, P, prompt, context, interval, flags):
    import torch
    from workload.driver import GpuRun
    wl = dataclasses.replace(QWEN3_8B_LAYER, num_q_heads=Hq, num_kv_heads=Hkv, page_size=P, beams=beams,
                             prompt_len=prompt, context=context, interval=interval, K=beams // 2, hidden=256)
    path = B.GB_PATH_AUTO if flags == "auto" else B.GB_PATH_GROUPED
    g, o = GpuRun(wl), OracleRun(wl, literal_kv=True)
    g.seed()
    o.seed()
    rounds = set(wl.rounds(include_final=True))
    step = 0
    while g.pos < wl.context:
        want = step % 9 == 0 or g.pos + 1 == wl.context or g.pos in rounds
        out = g.decode_step(path).cpu().numpy()
        for (layer, b), r in o.decode_step(compute=want).items():
            assert_rounded(out[layer, b], r, f"{flags}: attention L={o.pos} slot {b}")
        if g.pos in rounds:
            g.probe()
            o.probe()
            g.prune()
            o.prune()
            assert_pool_equal(g.pool.read_state(), o.pool, wl.page_size, means="tol", dtype="bf16")
        step += 1
    if beams > 2:                            # rows of released slots are zero, the others unchanged
        g.pool.release(torch.tensor([0, beams - 1], dtype=torch.int32, device="cuda"))
        out = g.decode_step(path).cpu().numpy()
        assert not out[:, [0, beams - 1]].any() and np.isfinite(out).all() and out[:, 1].any()
    assert g.pool.status() == 0
