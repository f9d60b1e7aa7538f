"""One-replica runs of a context that has its tables (k_run_r1 serves them for certain)
against the step kernels, bit for bit, and the run with which it gets them."""
import numpy as np
import pytest

import paper_2402_14718_gb300 as sb
from tests import inputs
from tests import test_gpu_run1 as run1

pytestmark = pytest.mark.gpu


def _build(ctx):
    for _ in range(3):
        run1._run(ctx, "bsb", 700, -1)
    assert sb.sb_step_kernels(ctx) == "k_run_r1"


def _same(ctx, variant, steps):
    a = run1._run(ctx, variant, steps, -1)
    assert sb.sb_step_kernels(ctx) == "k_run_r1"
    b = run1._run(ctx, variant, steps, 0)
    assert sb.sb_step_kernels(ctx) == "k_step_r1"
    assert np.isfinite(b[0]).all()
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])


@pytest.mark.parametrize("n", [1, 2, 3, 5, 31, 33, 127, 129, 500, 1023, 4099])
def test_small_problems(n):
    q = run1._sparse(n, 8, n) if n > 3 else (np.zeros(n + 1, np.int32), np.zeros(0, np.int32),
                                            np.zeros(0), np.full(n, 0.1))
    for prec in (sb.SB_J_FP32, sb.SB_J_BF16):
        ctx = sb.sb_create(n, *q, prec)
        _build(ctx)
        for variant in ("asb", "bsb", "dsb"):
            for steps in (16, 41):
                _same(ctx, variant, steps)


@pytest.mark.parametrize("n,per_row", [(20000, 12), (40001, 30), (130000, 6)])
def test_larger_problems(n, per_row):
    ctx = sb.sb_create(n, *run1._sparse(n, per_row, 3), sb.SB_J_BF16)
    _build(ctx)
    for variant in ("bsb", "dsb"):
        _same(ctx, variant, 33)


def test_batch_and_new_weights():
    ctx = sb.sb_create_batch([run1._sparse(n, 10, n) for n in (300, 37, 1500)])
    _build(ctx)
    _same(ctx, "bsb", 40)
    q = inputs.random_qubo(400, 12, 3)
    ctx = sb.sb_create(q.n, q.rowptr, q.col, q.val, q.lin)
    _build(ctx)
    _same(ctx, "bsb", 30)
    sb.sb_set_weights(ctx, (q.val > 0).astype(np.int8), np.abs(q.lin), 0.5, 0.7)
    _same(ctx, "bsb", 30)


def test_the_run_that_pays_for_the_tables():
    """A new context's short run takes the step kernels, as one without tables always did;
    a long one builds them at once, and so does the last of several short ones."""
    n = 20000
    q = run1._sparse(n, 12, 3)
    ctx = sb.sb_create(n, *q, sb.SB_J_BF16)
    run1._run(ctx, "bsb", 20, -1)
    assert sb.sb_step_kernels(ctx).startswith("k_step_r1")
    k = 1
    while sb.sb_step_kernels(ctx) != "k_run_r1" and k < 60:
        run1._run(ctx, "bsb", 20, -1)
        k += 1
    assert 5 < k < 60
    ctx = sb.sb_create(n, *q, sb.SB_J_BF16)
    run1._run(ctx, "bsb", 1000, -1)
    assert sb.sb_step_kernels(ctx) == "k_run_r1"
