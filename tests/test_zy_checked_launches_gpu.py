"""The checked build on launches of several iterations: items beyond the cached
ones, short items, restart with per-item extrapolation indices, rings shorter
than a launch, batches, and the planned steps of the unrolled solve and of its
adjoint (every plan, item, sum and history index verified on the device)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_index_checks_of_launches():
    cmd = [sys.executable, "-m", "pytest", "-q", "-x", "-p", "no:cacheprovider", "tests/test_step_launch_gpu.py",
           "tests/test_step_last_sums_gpu.py", "tests/test_step_record_interval_gpu.py",
           "tests/test_gpu_parity.py::test_unrolled_context_reuse_with_new_lambdas"]
    res = subprocess.run(cmd, cwd=ROOT, env=dict(os.environ, SPG_CHECKED="1"), capture_output=True, text=True, timeout=1800)
    tail = (res.stdout + res.stderr)[-3000:]
    print(tail)
    assert res.returncode == 0, tail
    assert "passed" in res.stdout and "SPG_ECHECK" not in res.stdout
