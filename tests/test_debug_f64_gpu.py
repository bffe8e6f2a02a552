"""The bounds-checking build on the binary64 tensor-core and unaligned kernels
(tests/debug_build_f64_cases.py): no address outside its operand."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def test_binary64_and_unaligned_cases_under_bounds_checks():
    pytest.importorskip("torch")
    sys.path.insert(0, ROOT)
    from paper_2002_03258_gb300 import build as b
    b.build(debug=True)
    r = subprocess.run([sys.executable, os.path.join(HERE, "debug_build_f64_cases.py")], env=dict(os.environ, TSM2_DEBUG="1"),
                       cwd=ROOT, capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-3000:]
    assert "DEBUG-F64-OK" in r.stdout, r.stdout[-2000:]
