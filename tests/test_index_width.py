"""Grid-stride loops over the stencils: N goes up to 2^31 - 1, so the index may
pass it by a stride before the loop ends and must not be a signed 32-bit one
(a negative index would pass `node < N` and address memory before the arrays)."""

import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_stencil_loops_do_not_overflow():
    loops = []
    for f in ("weights.cu", "refined.cu"):
        with open(os.path.join(ROOT, "paper_2107_03632_gb300", "csrc", f)) as src:
            loops += re.findall(r"for \((\w+) node = blockIdx[^;]*;([^;]*);", src.read())
    assert loops
    for kind, cond in loops:
        assert kind in ("unsigned", "int64_t") and "(unsigned)N" in cond, (kind, cond)
