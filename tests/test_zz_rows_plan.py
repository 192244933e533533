"""The work plan that gb_paged_decode_noalloc's kernel makes for itself: one to four rows per thread,
rows that cannot be read (their output zero, the status of that call only), and the
merge of the rest by the second launch.  Tolerance as in test_zz_no_alloc_sizes (fp32 sums against fp64)."""
import numpy as np
import pytest

from tests.test_zz_no_alloc_sizes import _setup

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,rows,longest", [("f32", 255, 40), ("bf16", 256, 17), ("f32", 257, 300),
                                                ("bf16", 1024, 60), ("f32", 1023, 20), ("bf16", 24, 5000)])
def test_rows_that_cannot_be_read(cuda, dtype, rows, longest):
    import torch
    from paper_2608_08020_gb300 import binding as B
    rng = np.random.default_rng(rows)
    lens = rng.integers(0, longest + 1, rows)
    lens[-1] = longest
    args = (dtype, 4, 2, 16, lens.tolist())
    call, ref = _setup(*args, seed=rows)
    bad = sorted({0, rows // 2, rows - 1})
    good0 = call()
    assert B.gb_paged_decode_noalloc_status() == 0
    t = next(c.cell_contents for c in call.__closure__ if isinstance(c.cell_contents, dict))
    keep = t["lens"].clone()
    for n, b in enumerate(bad):
        t["lens"][b] = -3 if n % 2 else 16 * t["tables"].shape[1] + 1
    out = call()
    assert B.gb_paged_decode_noalloc_status() == B.GB_ERR_INVALID
    want = ref.clone()
    want[bad] = 0
    assert bool(((out.double() - want).abs() <= 1e-5 * (1 + want.abs())).all())
    assert not bool(out[bad].any())
    t["lens"].copy_(keep)
    again = call()
    assert B.gb_paged_decode_noalloc_status() == 0
    assert torch.equal(again, good0)
