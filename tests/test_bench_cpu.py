"""What the benchmark reports of launches that take several steps (no GPU)."""
import os
import re
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_bytes_of_launches_that_take_several_steps():
    sys.path.insert(0, ROOT)
    import bench
    # 400 steps, 3 per launch: 134 launches a pass, the last of one step
    n, b = bench.launches_and_bytes([400], 100, 3, "velocity", "superposition", False)
    assert (n, b) == (268, 134 * 100 * (28 + 28))
    n, b = bench.launches_and_bytes([10, 4], 100, 4, "density", "symmetric", True)
    assert (n, b) == (8, 4 * 100 * ((16 + 8) + (32 + 8 + 16)))
    n, b = bench.launches_and_bytes([5], 100, 1, "velocity", "reverse", True)   # no compensation in this mode
    assert (n, b) == (10, 5 * 100 * ((16 + 4) + (32 + 4 + 8)))


def test_timed_launches_overlap_as_a_users_do():
    # events between the launches of a pass keep them apart; the timed calls have
    # none where launches take several steps
    text = open(os.path.join(ROOT, "bench.py")).read()
    assert "events = steps_per_launch == 1" in text
    timed = text[text.index("events = steps_per_launch == 1"):text.index("clk = clocks.stop()")]
    assert re.findall(r"timing_enable\((\w+)\)", timed) == ["events", "events"]


@pytest.mark.gpu
def test_bench_names_the_kernel_of_2d_workloads():
    import json
    import subprocess
    r = subprocess.run([sys.executable, os.path.join(ROOT, "bench.py"), "--workload", "w0", "--steps", "3", "--warmup",
                        "3", "--no-e2e", "--no-cpu-baseline"], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    roof = json.loads(r.stdout.strip().splitlines()[-1])["roofline"]
    assert roof["kernel"] == "step2d_tile" and roof["steps_per_launch"] > 1 and roof["bound"] == "issue"
    assert 0 < roof["frac"] < 1
