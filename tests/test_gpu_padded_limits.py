"""Padded replica counts where device memory runs short, readout buffers that are
no memory of the context's device, and one-replica runs under capture: what runs
without padding, copies or tables runs with them too, with the same results."""
import ctypes

import numpy as np
import pytest

import paper_2402_14718_gb300 as sb
from tests import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("spare", [256, 320])
def test_padded_state_or_its_sign_bytes_do_not_fit(spare):
    """400,000 rows at 50 replicas: 229 MiB of state as given, 293 MiB padded, 342 MiB
    with the sign bytes; `spare` MiB are left, so the state, then the bytes, do not fit."""
    import torch
    n, R, mb = 400000, 50, 1 << 20
    i = np.arange(n)
    col = np.sort((i[:, None] + np.array([-7, -1, 1, 7])) % n, axis=1).ravel().astype(np.int32)
    args = (n, (4 * np.arange(n + 1)).astype(np.int32), col, np.ones(4 * n), np.full(n, 0.3))
    rng = np.random.default_rng(2)
    x = rng.uniform(-1, 1, size=(n, R)).astype(np.float32)
    y = rng.uniform(-0.3, 0.3, size=(n, R)).astype(np.float32)
    sched = torch.linspace(0.2, 0.6, 5, device="cuda")

    def go(ctx):
        sb.sb_set_state(ctx, x, y)
        sb.sb_advance(ctx, "dsb", 1.0, 0.3, 0.4, 5, sched)
        return sb.sb_get_state(ctx)

    ctx = sb.sb_create(*args)
    want = go(ctx)
    sb.sb_destroy(ctx)
    ctx = sb.sb_create(*args)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    fill = torch.empty(free - spare * mb, dtype=torch.uint8, device="cuda")
    try:
        got = go(ctx)
    finally:
        del fill
        torch.cuda.empty_cache()
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])


def test_readout_into_pinned_host_memory():
    import torch
    q = inputs.random_qubo(300, 9, 5)
    ctx = sb.sb_create(q.n, q.rowptr, q.col, q.val, q.lin)
    sb.sb_run(ctx, "bsb", 1.0, 0.3, 0.4, 20, 8, seed=3)
    E = torch.empty((1, 8), dtype=torch.float64, device="cuda")
    b, r = torch.empty(1, dtype=torch.float64, device="cuda"), torch.empty(1, dtype=torch.int32, device="cuda")
    sb.sb_readout_device(ctx, E, b, r)
    torch.cuda.synchronize()
    Eh, bh, rh = (torch.empty_like(t, device="cpu").pin_memory() for t in (E, b, r))
    sb._lib.check(sb.lib.sb_readout_device(ctx.handle, *(ctypes.c_void_p(t.data_ptr()) for t in (Eh, bh, rh)),
                                           None, None))
    torch.cuda.synchronize()
    assert torch.equal(Eh, E.cpu()) and torch.equal(bh, b.cpu()) and torch.equal(rh, r.cpu())


@pytest.mark.parametrize("before", [4, 20])
def test_one_replica_run_under_capture(before):
    """Captured after a run too short for the run's tables, and after one with them."""
    import torch
    q = inputs.random_qubo(700, 9, 5)
    rng = np.random.default_rng(2)
    x = rng.uniform(-1, 1, size=(700, 1)).astype(np.float32)
    sched = torch.linspace(0.2, 0.6, 24, device="cuda")
    ctx = sb.sb_create(q.n, q.rowptr, q.col, q.val, q.lin)
    stream = torch.cuda.Stream()

    def advance(steps):
        sb.sb_advance(ctx, "bsb", 1.0, 0.3, 0.4, steps, sched, stream=stream)

    sb.sb_set_option(ctx, sb.SB_OPT_R1_LANES, 0)
    sb.sb_set_state(ctx, x, x)
    advance(24)
    want = sb.sb_get_state(ctx)
    sb.sb_set_option(ctx, sb.SB_OPT_R1_LANES, -1)
    advance(before)
    stream.synchronize()
    sb.sb_set_state(ctx, x, x)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream, capture_error_mode="thread_local"):
        advance(24)
    g.replay()
    got = sb.sb_get_state(ctx)
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
