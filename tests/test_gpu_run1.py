"""One-replica runs in one launch (k_run_r1) against the step kernels
(SB_OPT_R1_LANES set), bit for bit: sizes at the edges of the row chunks and
slices, empty and dense rows, odd and even step counts, batches, weights."""
import numpy as np
import pytest

import paper_2402_14718_gb300 as sb
from tests import inputs

pytestmark = pytest.mark.gpu


def _run(ctx, variant, steps, lanes, c0=0.4):
    sb.sb_set_option(ctx, sb.SB_OPT_R1_LANES, lanes)
    sb.sb_run(ctx, variant, 1.0, c0, 0.3, steps, 1, seed=7)
    return sb.sb_get_state(ctx)


def _same(ctx, variant, steps):
    a, b = _run(ctx, variant, steps, -1), _run(ctx, variant, steps, 0)
    assert np.isfinite(b[0]).all()
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])


def _sparse(n, per_row, seed):
    """Random symmetric pattern, row 0 joined to up to 700 rows, row 1 empty."""
    rng = np.random.default_rng(seed)
    i = rng.integers(0, n, size=n * per_row // 2)
    j = rng.integers(0, n, size=len(i))
    hub = rng.choice(n, size=min(n, 700), replace=False)
    i, j = np.concatenate([i, np.zeros(len(hub), int)]), np.concatenate([j, hub])
    ok = (i != j) & (i != 1) & (j != 1)
    key = np.unique(np.minimum(i, j)[ok] * n + np.maximum(i, j)[ok])
    i, j = key // n, key % n
    v = rng.choice([-1.0, 1.0, 0.3], size=len(i)) * 0.2
    r, c, v = np.concatenate([i, j]), np.concatenate([j, i]), np.concatenate([v, v])
    o = np.lexsort((c, r))
    rowptr = np.concatenate([[0], np.cumsum(np.bincount(r, minlength=n))]).astype(np.int32)
    return rowptr, c[o].astype(np.int32), v[o], rng.uniform(0, 0.2, n)


@pytest.mark.parametrize("n", [1, 2, 3, 5, 31, 33, 127, 129, 500, 1023, 4099])
@pytest.mark.parametrize("variant", ["asb", "bsb", "dsb"])
def test_small_problems(n, variant):
    q = _sparse(n, 8, n) if n > 3 else (np.zeros(n + 1, np.int32), np.zeros(0, np.int32),
                                       np.zeros(0), np.full(n, 0.1))
    for prec in (sb.SB_J_FP32, sb.SB_J_BF16):
        ctx = sb.sb_create(n, *q, prec)
        for steps in (16, 41):
            _same(ctx, variant, steps)


@pytest.mark.parametrize("n,per_row", [(20000, 12), (40001, 30), (130000, 6)])
@pytest.mark.parametrize("variant", ["bsb", "dsb"])
def test_larger_problems_and_resumed_runs(n, per_row, variant):
    ctx = sb.sb_create(n, *_sparse(n, per_row, 3), sb.SB_J_BF16)
    _same(ctx, variant, 33)
    # a second run on the same tables, resumed after an odd number of steps
    import torch
    sched = torch.linspace(0.3, 0.6, 17, device="cuda")
    out = []
    for lanes in (-1, 0):
        x, y = _run(ctx, variant, 21, lanes)
        sb.sb_advance(ctx, variant, 1.0, 0.4, 0.3, 17, sched)
        out.append(sb.sb_get_state(ctx))
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])


def test_batch_and_new_weights():
    qs = [_sparse(n, 10, n) for n in (300, 37, 1500)]
    ctx = sb.sb_create_batch(qs)
    _same(ctx, "bsb", 40)
    q = inputs.random_qubo(400, 12, 3)
    ctx = sb.sb_create(q.n, q.rowptr, q.col, q.val, q.lin)
    _same(ctx, "bsb", 30)
    sb.sb_set_weights(ctx, (q.val > 0).astype(np.int8), np.abs(q.lin), 0.5, 0.7)
    _same(ctx, "bsb", 30)
