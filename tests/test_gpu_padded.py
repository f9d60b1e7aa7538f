"""Replica counts that are no multiple of 4 (stored in padded rows) and the
step kernel's neighbour batches: every replica must come out as it does in a run
of another replica count, bit for bit, and states must pass in and out whole."""
import numpy as np
import pytest

import paper_2402_14718_gb300 as sb
from tests import inputs

pytestmark = pytest.mark.gpu


def _ctx(n, degree, seed, prec):
    q = inputs.random_qubo(n, degree, seed)
    return sb.sb_create(n, q.rowptr, q.col, q.val, q.lin, prec)


def _advance(ctx, variant, x, y, steps, on_device=False):
    import torch
    if on_device:
        x, y = torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda()
    sb.sb_set_state(ctx, x, y)
    sched = torch.tensor(np.linspace(0.2, 0.6, steps).astype(np.float32), device="cuda")
    sb.sb_advance(ctx, variant, 1.0, 0.3, 0.4, steps, sched)
    return sb.sb_get_state(ctx)


@pytest.mark.parametrize("R", [2, 3, 5, 7, 13, 30, 33, 50, 63, 65, 95, 127, 130, 250])
@pytest.mark.parametrize("variant", ["asb", "bsb", "dsb"])
def test_padded_rows_give_the_same_replicas(R, variant):
    n = 257
    rng = np.random.default_rng(R)
    x = rng.uniform(-1, 1, size=(n, R)).astype(np.float32)
    y = rng.uniform(-0.3, 0.3, size=(n, R)).astype(np.float32)
    x[rng.random(x.shape) < 0.02] = 0.0
    ctx = _ctx(n, 9, 5, sb.SB_J_BF16)
    sb.sb_set_state(ctx, x, y)
    x0, y0 = sb.sb_get_state(ctx)
    assert np.array_equal(x0, x) and np.array_equal(y0, y)
    xa, ya = _advance(ctx, variant, x, y, 5, on_device=R % 2 == 1)
    E = sb.sb_energy(ctx, None, R)
    T, Eb, rb = sb.sb_best(ctx)
    # one replica at a time: the one-replica kernels, same order of operations
    one = _ctx(n, 9, 5, sb.SB_J_BF16)
    for r in sorted({0, R // 2, R - 1}):
        xr, yr = _advance(one, variant, x[:, r:r + 1].copy(), y[:, r:r + 1].copy(), 5)
        assert np.array_equal(xr[:, 0], xa[:, r]) and np.array_equal(yr[:, 0], ya[:, r])
        assert np.allclose(sb.sb_energy(one, None, 1)[0, 0], E[0, r], rtol=1e-12)
    assert np.array_equal(T, (xa[:, rb[0]] > 0).astype(np.uint8)) and Eb[0] == E[0].min()


@pytest.mark.parametrize("prec", [sb.SB_J_FP32, sb.SB_J_BF16])
@pytest.mark.parametrize("n,R", [(40, 4), (40, 20), (40, 64), (9000, 20), (9000, 64), (40000, 64),
                                 (40000, 96), (5000, 512)])
def test_neighbour_batches_at_every_remainder(n, R, prec):
    """Row degrees 0 .. 39 (every remainder of the batches of 2, 4 and 8), on each
    side of the rules on spins, against one replica alone."""
    rng = np.random.default_rng(n + R)
    deg = np.arange(n) % 40
    pairs = set()
    for i in rng.choice(n, size=min(n, 400), replace=False):
        for j in rng.choice(n, size=min(int(deg[i]), n - 1), replace=False):
            if i != j:
                pairs.add((min(i, j), max(i, j)))
    ij = np.array(sorted(pairs))
    rows = np.concatenate([ij[:, 0], ij[:, 1]])
    cols = np.concatenate([ij[:, 1], ij[:, 0]])
    val = rng.choice([-1.0, 1.0, 0.5], size=len(ij))
    val = np.concatenate([val, val])
    o = np.lexsort((cols, rows))
    rowptr = np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=n))]).astype(np.int32)
    args = (n, rowptr, cols[o].astype(np.int32), val[o], rng.uniform(0, 1, n), prec)
    x = rng.uniform(-1, 1, size=(n, R)).astype(np.float32)
    y = rng.uniform(-0.3, 0.3, size=(n, R)).astype(np.float32)
    ctx, one = sb.sb_create(*args), sb.sb_create(*args)
    for variant in ("bsb", "dsb"):
        xa, ya = _advance(ctx, variant, x, y, 3)
        for r in (0, R - 1):
            xr, yr = _advance(one, variant, x[:, r:r + 1].copy(), y[:, r:r + 1].copy(), 3)
            assert np.array_equal(xr[:, 0], xa[:, r]) and np.array_equal(yr[:, 0], ya[:, r])
