"""The FP32 products on the tensor cores in the bounds-checking debug build; see
tests/bounds_debug_f32tc_check.py, which runs in a child process."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_no_access_outside_the_operands():
    from paper_2008_13145_gb300 import build
    build.build_debug_library()
    r = subprocess.run([sys.executable, os.path.join(ROOT, "tests", "bounds_debug_f32tc_check.py")],
                       env={**os.environ, "KSELECT_DEBUG_BOUNDS": "1"}, capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stderr[-3000:]
    res = json.loads(r.stdout.strip().splitlines()[-1])
    assert res["cases"] == 144 and res["handle_splits"] > 1, res
    assert res["out_of_bounds"] == 0, res
    assert res["worst_error_ratio"] <= 1e-5, res  # the library's FP32 tolerance
    assert all(n > 0 for n in res["flagged"]), res
