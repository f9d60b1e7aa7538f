"""sb_autotune of one replica: the one-launch run is a candidate like the others,
timed with its tables in place, and keeps its place where it is the fastest."""
import numpy as np
import pytest

import paper_2402_14718_gb300 as sb
from tests import test_gpu_run1 as run1

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,per_row", [(700, 8), (4099, 8), (20000, 30)])
@pytest.mark.parametrize("trial_steps", [1, 20, 50])
def test_one_replica_keeps_the_one_launch_run(n, per_row, trial_steps):
    """It takes half a step kernel's time or less at these sizes, however short the trial."""
    ctx = sb.sb_create(n, *run1._sparse(n, per_row, 3), sb.SB_J_BF16)
    cfg, us = sb.sb_autotune(ctx, "bsb", 1, trial_steps)
    assert cfg["rows_per_cta"] == cfg["l2_persist"] == cfg["tile"] == 0 and cfg["groups"] == 1
    a = run1._run(ctx, "bsb", 33, -1)
    assert sb.sb_step_kernels(ctx) == "k_run_r1"
    b = run1._run(ctx, "bsb", 33, 0)
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
