"""The bounded waits of the one-replica run (k_run_r1): a position that is never
published ends the run within SB_OPT_WAIT_NS, the next synchronising call says
so once, and the context runs on."""
import time

import numpy as np
import pytest

import paper_2402_14718_gb300 as sb
from tests import test_gpu_run1 as run1

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [31, 700, 20000])
@pytest.mark.parametrize("step", [0, 5])
def test_wait_runs_out(n, step):
    ctx = sb.sb_create(n, *run1._sparse(n, 12, 3), sb.SB_J_FP32)
    for _ in range(50):  # however many steps the tables are worth, these are enough
        good = run1._run(ctx, "bsb", 40, -1)
    assert sb.sb_step_kernels(ctx) == "k_run_r1"
    sb.sb_set_option(ctx, sb.SB_OPT_WAIT_NS, 1_000_000)
    sb.sb_set_option(ctx, sb.SB_OPT_TEST_SKIP_STAGE, step)
    t = time.perf_counter()
    with pytest.raises(sb.SbError, match="neighbour's position") as e:
        run1._run(ctx, "bsb", 40, -1)
    assert e.value.code == sb._lib.SB_ERR_TIMEOUT
    # 1 ms, where the default limit of 2 s would pass first
    assert time.perf_counter() - t < 1.0
    sb.sb_set_option(ctx, sb.SB_OPT_TEST_SKIP_STAGE, -1)
    sb.sb_set_option(ctx, sb.SB_OPT_WAIT_NS, 2_000_000_000)
    again = run1._run(ctx, "bsb", 40, -1)
    assert sb.sb_step_kernels(ctx) == "k_run_r1"
    assert np.array_equal(again[0], good[0]) and np.array_equal(again[1], good[1])
