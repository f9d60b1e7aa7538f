"""Which kernels serve a run (sb_step_kernels): the bit-for-bit comparisons of the
other tests compare what they mean to compare only while these hold."""
import numpy as np
import pytest

import paper_2402_14718_gb300 as sb
from tests import test_gpu_run1 as run1
from tests.test_gpu_factor_blocks import _grouped

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,per_row,one", [(31, 8, True), (4099, 8, True), (20000, 12, True),
                                           (40001, 30, True), (130000, 6, True),
                                           (60000, 100, False), (160000, 2, False)])
def test_one_replica(n, per_row, one):
    """The sizes of the one-replica tests, one whose couplings do not fit in shared
    memory (152 SMs of 220 KB hold 5.7 M of them at most), one with more rows than threads."""
    ctx = sb.sb_create(n, *run1._sparse(n, per_row, 3), sb.SB_J_BF16)
    for _ in range(50):  # however many steps the tables are worth, these are enough
        run1._run(ctx, "bsb", 33, -1)
    names = sb.sb_step_kernels(ctx)
    assert (names == "k_run_r1") == one and (one or names.startswith("k_step_r1"))
    run1._run(ctx, "bsb", 8, -1)
    assert sb.sb_step_kernels(ctx).startswith("k_step_r1")
    run1._run(ctx, "bsb", 33, 0)
    assert sb.sb_step_kernels(ctx) == "k_step_r1"


def test_replica_counts_and_options():
    q, member, couple = _grouped((3, 8, 40, 130), 3, 1)
    ctx = sb.sb_create(len(q[3]), *q, sb.SB_J_BF16)
    assert sb.sb_step_kernels(ctx) == ""

    def names(variant, R, fac=0, **opts):
        for k, v in opts.items():
            sb.sb_set_option(ctx, getattr(sb, k), v)
        sb.sb_set_option(ctx, sb.SB_OPT_FACTOR, fac)
        sb.sb_run(ctx, variant, 1.0, 0.05, 0.5, 3, R, seed=1)
        return sb.sb_step_kernels(ctx)

    sb.sb_set_factor(ctx, 4, member, couple, 1.0)
    assert names("dsb", 64, -1) == names("dsb", 50, -1) == "k_fac_sum_sgn + k_step_fac_sgn"
    assert names("bsb", 128, -1) == "k_fac_sum + k_step_rw"
    assert names("asb", 16, -1) == "k_fac_sum + k_step_fac"
    assert names("bsb", 50, -1) == names("dsb", 64) == "k_step"
    assert names("bsb", 256) == "k_step_rw"
    assert names("bsb", 64, SB_OPT_STREAM=1) == "k_step_stream"
    assert names("bsb", 64, SB_OPT_STREAM=0, SB_OPT_TILED=1) == "k_step_tiled"
    big = 40000
    ctx = sb.sb_create(big, *run1._sparse(big, 4, 3), sb.SB_J_BF16)
    sb.sb_run(ctx, "dsb", 1.0, 0.05, 0.5, 3, 64, seed=1)
    assert sb.sb_step_kernels(ctx) == "k_step_dsb16"


@pytest.mark.parametrize("rpc,R,kernel", [(0, 128, "k_step"), (32, 128, "k_step_dsb16"), (32, 64, "k_step"),
                                          (64, 64, "k_step_dsb16"), (64, 32, "k_step"), (0, 256, "k_step_dsb16")])
def test_dsb_rows_per_cta(rpc, R, kernel):
    """1.4 M spins at R = 128: more than two rows to a lane group take the other kernel."""
    n = 11000
    q = run1._sparse(n, 8, 3)
    ctx = sb.sb_create(n, *q, sb.SB_J_BF16)
    out = []
    for v in (rpc, 0):
        sb.sb_set_option(ctx, sb.SB_OPT_STEP_RPC, v)
        sb.sb_run(ctx, "dsb", 1.0, 0.4, 0.3, 5, R, seed=2)
        out.append((sb.sb_step_kernels(ctx),) + sb.sb_get_state(ctx))
    assert out[0][0] == kernel
    assert np.array_equal(out[0][1], out[1][1]) and np.array_equal(out[0][2], out[1][2])
