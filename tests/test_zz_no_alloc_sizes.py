"""gb_paged_decode_noalloc over the shares its warps take (one chunk, longer ones for few long rows,
even shares), each call twice and different sizes interleaved, so that a call finds the plan and the
records another size left.

fp32 and bf16 pages, probabilities in fp32: 1e-5 of the output's scale (fp32 sums), against fp64."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CASES = [  # dtype, G, Hkv, P, row lengths
    ("bf16", 4, 1, 16, [1]),                          # one pair, one chunk
    ("f32", 2, 2, 32, [15, 16, 17, 0, 33]),           # chunk edges, an empty row
    ("bf16", 8, 2, 64, [700, 1, 256, 129]),           # a few ragged rows
    ("f32", 4, 8, 16, [5000, 3]),                     # one long row: many records of a pair, longer shares
    ("bf16", 2, 8, 16, list(range(1, 301))),          # 2400 pairs: a warp takes several
    ("bf16", 4, 8, 32, [3000, 4096, 1, 2500] * 12),   # even shares
    ("f32", 8, 4, 64, [900 + 7 * i for i in range(90)]),
]


def _setup(dtype, G, Hkv, P, lens, seed):
    import torch
    from paper_2608_08020_gb300 import binding as B
    dt, D = (torch.bfloat16, 128) if dtype == "bf16" else (torch.float32, 64)
    g = torch.Generator(device="cuda").manual_seed(seed)
    lens = np.array(lens, np.int32)
    width = -(-int(lens.max()) // P)
    num = int((-(-lens // P)).sum()) + 3
    ids = np.random.default_rng(seed).permutation(num).astype(np.int32)
    tables, at = np.zeros((len(lens), width), np.int32), 0
    for b, n in enumerate(-(-lens // P)):
        tables[b, :n] = ids[at:at + n]
        at += n
    t = dict(kv=torch.randn(num, 2, Hkv, P, D, generator=g, device="cuda").to(dt), tables=torch.from_numpy(tables).cuda(),
             lens=torch.from_numpy(lens).cuda(), q=torch.randn(len(lens), G * Hkv, D, generator=g, device="cuda").to(dt))
    ref = torch.zeros(len(lens), G * Hkv, D, dtype=torch.float64, device="cuda")
    for b, n in enumerate(lens):
        if n:
            pages = t["kv"][t["tables"][b, :-(-int(n) // P)].long()]
            k, v = (pages[:, w].permute(1, 0, 2, 3).reshape(Hkv, -1, D)[:, :int(n)].double() for w in (0, 1))
            s = torch.bmm(t["q"][b].double().view(Hkv, G, D), k.transpose(1, 2)) / math.sqrt(D)
            ref[b] = torch.bmm(torch.softmax(s, -1), v).reshape(-1, D)

    def call():
        out = torch.full(ref.shape, float("nan"), dtype=torch.float32, device="cuda")
        B.gb_paged_decode_noalloc(B.GbPagedDecodeArgs(
            t["kv"].data_ptr(), t["tables"].data_ptr(), t["lens"].data_ptr(), t["q"].data_ptr(), out.data_ptr(),
            len(lens), G * Hkv, Hkv, D, P, B.GB_BF16 if dtype == "bf16" else B.GB_F32, width, num, 1 / math.sqrt(D)))
        return out
    return call, ref


def test_sizes_interleaved(cuda):
    from paper_2608_08020_gb300 import binding as B
    made = [_setup(*c, seed=i) for i, c in enumerate(CASES)]
    for order in (range(len(made)), reversed(range(len(made)))):
        for i in order:
            call, ref = made[i]
            outs = [call(), call()]
            assert B.gb_paged_decode_noalloc_status() == 0
            for out in outs:
                err = (out.double() - ref).abs()
                assert bool((err <= 1e-5 * (1 + ref.abs())).all()), (CASES[i][:4], float(err.max()))
