"""Every store to an operand or to the workspace in the binary64 and unaligned
kernels stands behind a bounds check of the debug build (common.cuh)."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2002_03258_gb300", "csrc")
STORE = re.compile(r"\bC\[[^;=]*\] = |__stcg\(|\bput\(dst|^\s*\*dst = ")


@pytest.mark.parametrize("name,least", [("tsm2_f64tc.cu", 7), ("tsm2_f64s.cu", 3), ("tsm2_shift.cu", 3)])
def test_stores_are_checked(name, least):
    with open(os.path.join(CSRC, name)) as f:
        lines = f.read().split("\n")
    stores = [i for i, line in enumerate(lines) if STORE.search(line) and not line.lstrip().startswith("//")]
    assert len(stores) >= least, "the pattern no longer finds the stores"
    for i in stores:
        above = lines[max(0, i - 16):i + 1]
        assert any("dbg_" in line for line in above), f"{name}:{i + 1}: {lines[i].strip()}"
