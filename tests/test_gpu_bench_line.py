"""The benchmark's output: one line that carries the headline and is short enough for a log that keeps the end of it."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_default_run_prints_one_short_line():
    import bench
    r = subprocess.run([sys.executable, "bench.py", "--steps", "3", "--warmup", "3"], cwd=ROOT, capture_output=True, text=True, timeout=600, check=True)
    lines = [x for x in r.stdout.splitlines() if x.strip()]
    assert len(lines) == 1 and len(lines[0]) <= bench.LINE_BYTES, (len(lines), len(r.stdout))
    out = json.loads(lines[0])
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling", "vs_baseline", "dtype", "data", "config",
                "e2e", "gpu_launches", "clocks", "roofline", "cpu_baseline"):
        assert key in out, key
    assert out["value"] > 0 and out["e2e"]["value"] > 0 and out["e2e"]["h2d_bytes_per_step"] > 0 and out["e2e"]["d2h_bytes_per_step"] > 0
    assert out["config"]["workload"] == bench.DEFAULT_WORKLOAD and out["steps"] == 3 and out["warmup"] == 3
