"""The debug-bounds build (see test_debug_bounds_gpu.py) on the kernels that
set-up picks by itself: register sweeps, column-tiled transfers, the device's
coarse inverse and the coarse solve, forward and transposed, record no index
outside its array."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_debug_build_records_nothing_on_the_chosen_sweeps(cuda):
    from paper_2605_21046_gb300 import build
    build.build(debug_bounds=True)
    env = dict(os.environ, SG_DEBUG_BOUNDS="1")
    r = subprocess.run([sys.executable, os.path.join(ROOT, "tests", "_bounds_sweeps_worker.py")], env=env,
                       capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
    out = json.loads(r.stdout.strip().splitlines()[-1])
    assert out["library"] == "libsg_debug.so"
    for stage in ("after_sweeps", "after_long_rows", "after_coarse"):
        assert out[stage]["enabled"] == 1 and out[stage]["count"] == 0, (stage, out[stage])
