"""A handle call whose choice needs no scratch runs that choice when there is no memory for
the scratch of a split tensor-core product; the debug build makes the allocation fail
(tests/scratch_fallback_check.py, in a child process)."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_the_selected_config_runs_without_scratch():
    from paper_2008_13145_gb300 import build
    build.build_debug_library()
    r = subprocess.run([sys.executable, os.path.join(ROOT, "tests", "scratch_fallback_check.py")],
                       env={**os.environ, "KSELECT_DEBUG_BOUNDS": "1"}, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-3000:]
    res = json.loads(r.stdout.strip().splitlines()[-1])
    assert res["plan_splits"] > 1 and res["conv_splits"] > 1, res
    assert res["gemm_same_as_config"] and res["then_tensor_cores"], res
    assert max(res["errors"]) <= 1e-5, res  # the library's FP32 tolerance
    assert res["conv"][0] and not res["conv"][1] and res["conv"][2] <= 1e-4, res  # |x||w| is up to 50 times the result
    assert res["split_choice"] == -4, res


def test_release_builds_have_no_such_hook(lib):
    assert lib._lib.kselect_debug_fail_scratch(1) == -2
