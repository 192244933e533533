"""Which pointers the kernels may declare const __restrict__.  Launched programmatically a kernel may start
while its predecessor still writes, and const __restrict__ data may be read as constant for the kernel's
whole life: so only what the caller owns (weights, masks, hidden states), never what another kernel of
the library writes (queries, partial sums, activations, slot state)."""
import re
from pathlib import Path

CSRC = Path(__file__).resolve().parent.parent / "paper_2608_08020_gb300" / "csrc"
CALLERS = {
    "mlp.cu": {"b1", "w2", "mask"},
    "probe.cu": {"hidden", "w", "mask"},
    "scorer.cu": {"h", "g", "b", "w_out", "b_out"},
}


def test_only_the_callers_data_is_read_as_constant():
    seen = 0
    for f in sorted(CSRC.glob("*.cu*")):
        for m in re.finditer(r"const \w+\s*\*\s*__restrict__\s+(\w+)", f.read_text()):
            seen += 1
            assert m[1] in CALLERS.get(f.name, set()), f"{f.name}: {m[0]}"
    assert seen > 0
