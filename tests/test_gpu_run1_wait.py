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


@pytest.mark.parametrize("whole", [True, False])
def test_asynchronous_readout_of_a_run_that_gave_up(whole):
    """No host call has looked at the run when its energies are read: they are NaN."""
    import torch
    n = 700
    rowptr, col, val, lin = run1._sparse(n, 12, 3)
    ctx = sb.sb_create(n, rowptr, col, np.sign(val) if whole else val, lin, sb.SB_J_FP32)
    for _ in range(50):
        run1._run(ctx, "bsb", 40, -1)
    E, b = (torch.zeros(1, dtype=torch.float64, device="cuda") for _ in range(2))
    r = torch.full((1,), 7, dtype=torch.int32, device="cuda")
    T = torch.zeros(n, dtype=torch.uint8, device="cuda")

    def read(step):
        sb.sb_set_option(ctx, sb.SB_OPT_TEST_SKIP_STAGE, step)
        sb.sb_set_option(ctx, sb.SB_OPT_WAIT_NS, 1_000_000 if step >= 0 else 2_000_000_000)
        sb.sb_run(ctx, "bsb", 1.0, 0.4, 0.3, 40, 1, seed=7)
        assert sb.sb_step_kernels(ctx) == "k_run_r1"
        sb.sb_readout_device(ctx, E, b, r, T)
        torch.cuda.synchronize()
        return E.item(), b.item(), r.item()

    good = read(-1)
    assert np.isfinite(good[0]) and good[:1] == good[1:2] and good[2] == 0
    late = read(3)
    assert np.isnan(late[0]) and np.isnan(late[1]) and late[2] == 0
    with pytest.raises(sb.SbError, match="neighbour's position"):
        sb.sb_best(ctx)
    assert read(-1) == good
