"""The bench line's figures belong to the engine that its calls take without statistics."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("workload,engine", [("er1k", "columns"), ("rmat24 --scale 15", "passes")])
def test_timed_steps_run_in_the_engine_of_the_default_call(workload, engine):
    out = subprocess.run([sys.executable, "bench.py", "--workload", *workload.split(), "--steps", "3", "--warmup", "3",
                          "--no-cpu-baseline"], cwd=ROOT, capture_output=True, text=True, timeout=600)
    assert out.returncode == 0, out.stderr[-2000:]
    line = json.loads(out.stdout.strip().splitlines()[-1])
    assert line["config"]["engines"]["ic"] == engine
    assert ("column engine" in line["config"]["call_mode"]) == ("columns" in line["config"]["engines"].values())
    if engine == "columns":  # a launch a call, IC and LT
        assert line["gpu_launches"] == 6
    else:
        assert line["gpu_launches"] > 60
    for k in line["kernels"].values():  # event times from the pass engine either way
        assert k["expand_ms_per_step"] > 0 and k["edge_checks_per_step"] > 0
