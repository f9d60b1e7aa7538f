"""bench.py names the kernels that ran: its line against the library's own word for the
same workload, where the choice changed with sizes, forms and replica counts."""
import json
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("args,kernels,per_run", [
    (["--workload", "event100", "--sb-steps", "200"], "k_run_r1", 3 + 1 + 5),
    (["--workload", "event1000", "--variant", "dsb", "--sb-steps", "50"],
     "k_fac_sum_sgn + k_step_fac_sgn", 4 + 100 + 5),
    (["--workload", "event500", "--variant", "dsb", "--sb-steps", "50", "--no-factor"], "k_step",
     4 + 50 + 5),
])
def test_kernels_and_launches(args, kernels, per_run):
    r = subprocess.run([sys.executable, "bench.py", "--steps", "1", "--no-cpu-baseline", "--no-ttt",
                        "--no-energy-check", "--no-clocks"] + args, cwd=ROOT, capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    line = json.loads(r.stdout.strip().splitlines()[-1])
    assert line["roofline"]["kernel"] == kernels
    assert line["gpu_launches"] == per_run
