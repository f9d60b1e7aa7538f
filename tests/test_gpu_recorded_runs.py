"""Runs and readouts that a caller recorded into a CUDA graph, replayed after
sb_set_weights gave the context new couplings: they read the context's
couplings in place, so a replay gives what a fresh call gives."""
import numpy as np
import pytest

import paper_2402_14718_gb300 as sb
from tests import inputs
from tests import test_gpu_factor_blocks as blocks

pytestmark = pytest.mark.gpu


def _weights(ctx, q, w_c):
    sb.sb_set_weights(ctx, (q.val > 0).astype(np.int8), np.abs(q.lin), 0.5, w_c)


def _record(stream, f):
    import torch
    stream.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream, capture_error_mode="thread_local"):
        f()
    return g


@pytest.mark.parametrize("n", [33, 700, 1500])
@pytest.mark.parametrize("variant,prec", [("bsb", sb.SB_J_FP32), ("dsb", sb.SB_J_BF16)])
def test_one_replica_run(n, variant, prec):
    """The run's tables carry the couplings: new weights are filled in where they lie."""
    import torch
    q = inputs.random_qubo(n, 9, 5)
    x = np.random.default_rng(2).uniform(-1, 1, size=(n, 1)).astype(np.float32)
    sched = torch.linspace(0.2, 0.6, 24, device="cuda")
    ctx = sb.sb_create(q.n, q.rowptr, q.col, q.val, q.lin, prec)
    stream = torch.cuda.Stream()

    def advance():
        sb.sb_advance(ctx, variant, 1.0, 0.3, 0.4, 24, sched, stream=stream)

    def fresh():
        sb.sb_set_option(ctx, sb.SB_OPT_R1_LANES, 0)
        sb.sb_set_state(ctx, x, x)
        advance()
        out = sb.sb_get_state(ctx)
        sb.sb_set_option(ctx, sb.SB_OPT_R1_LANES, -1)
        return out

    _weights(ctx, q, 1.0)
    sb.sb_set_state(ctx, x, x)
    for _ in range(100):  # however many steps the tables are worth, these are enough
        advance()
    sb.sb_set_state(ctx, x, x)
    g = _record(stream, advance)
    seen = []
    for w_c in (1.0, 0.6, 2.0):
        _weights(ctx, q, w_c)
        want = fresh()
        sb.sb_set_state(ctx, x, x)
        g.replay()
        got = sb.sb_get_state(ctx)
        assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
        seen.append(got[0])
    assert not np.array_equal(seen[0], seen[1])


def _ring(n):
    """Rows joined to their neighbours at distance 1 (conflict) and 7 (consistent)."""
    i = np.arange(n)
    col = np.sort((i[:, None] + np.array([-7, -1, 1, 7])) % n, axis=1)
    gap = np.abs(col - i[:, None])
    cls = (np.minimum(gap, n - gap) == 1).astype(np.int8).ravel()
    return inputs.QuboArrays(n, (4 * np.arange(n + 1)).astype(np.int32), col.ravel().astype(np.int32),
                             np.where(cls, 1.0, -1.0), np.full(n, 0.3))


@pytest.mark.parametrize("n,R", [(700, 8), (700, 50), (40000, 64), (200000, 4)])
@pytest.mark.parametrize("first", [1.0, 0.6])
def test_readout(n, R, first):
    """Energies from selection bits need whole-number weights, which sb_set_weights
    takes and gives; a fresh readout of another context is the reference."""
    import torch
    q = _ring(n)
    ctx, other = (sb.sb_create(q.n, q.rowptr, q.col, q.val, q.lin) for _ in range(2))
    rng = np.random.default_rng(n + R)
    x = rng.uniform(-1, 1, size=(n, R)).astype(np.float32)
    E, want = (torch.zeros((1, R), dtype=torch.float64, device="cuda") for _ in range(2))
    b, r = torch.zeros(1, dtype=torch.float64, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    stream = torch.cuda.Stream()
    _weights(ctx, q, first)
    sb.sb_set_state(ctx, x, x)
    sb.sb_readout_device(ctx, E, b, r, stream=stream)
    g = _record(stream, lambda: sb.sb_readout_device(ctx, E, b, r, stream=stream))
    for w_c in (first, 0.6, 1.0, 0.37, 2.0, first):
        _weights(ctx, q, w_c)
        _weights(other, q, w_c)
        sb.sb_set_state(other, x, x)
        sb.sb_readout_device(other, want)
        sb.sb_readout_device(ctx, E, b, r)           # a fresh one, between two replays
        torch.cuda.synchronize()
        assert torch.allclose(E, want, rtol=1e-12, atol=0)
        E.zero_()
        torch.cuda.synchronize()
        g.replay()
        torch.cuda.synchronize()
        assert torch.allclose(E, want, rtol=1e-12, atol=0)
        assert b.item() == E.min().item() and r.item() == E.argmin().item()


@pytest.mark.parametrize("before,then", [(0.6, 1.0), (1.0, 0.6), (1.0, 1.0)])
def test_readout_recorded_right_after_new_weights(before, then):
    """Buffers made for other weights serve the recording: it makes none of its own."""
    import torch
    n, R = 3000, 8
    q = _ring(n)
    ctx = sb.sb_create(q.n, q.rowptr, q.col, q.val, q.lin)
    x = np.random.default_rng(1).uniform(-1, 1, size=(n, R)).astype(np.float32)
    E = torch.zeros((1, R), dtype=torch.float64, device="cuda")
    stream = torch.cuda.Stream()
    _weights(ctx, q, before)
    sb.sb_set_state(ctx, x, x)
    sb.sb_readout_device(ctx, E, stream=stream)
    _weights(ctx, q, then)
    g = _record(stream, lambda: sb.sb_readout_device(ctx, E, stream=stream))
    for w_c in (then, 1.0, 0.6, 1.0):
        _weights(ctx, q, w_c)
        g.replay()
        torch.cuda.synchronize()
        got = E.cpu().numpy()
        assert np.allclose(got, sb.sb_energy(ctx, None, R), rtol=1e-12, atol=0)


@pytest.mark.parametrize("variant", ["dsb", "bsb", "asb"])
@pytest.mark.parametrize("R", [6, 50, 127])
@pytest.mark.parametrize("warm", [False, True])
def test_padded_run(variant, R, warm):
    """Replica counts that are stored padded, with a factor set, recorded before any other
    run of the context or after one: the recorded run takes what the kernels for the
    count itself took, the CSR, and outlives the factor and the weights."""
    import torch
    q, member, couple = blocks._grouped((3, 8, 40, 130), 3, 1)
    n = len(q[3])
    rng = np.random.default_rng(R)
    x = rng.uniform(-1, 1, size=(n, R)).astype(np.float32)
    y = rng.uniform(-0.3, 0.3, size=(n, R)).astype(np.float32)
    sched = torch.linspace(0.2, 0.6, 4, device="cuda")
    dt = 0.1 if variant == "asb" else 0.4
    stream = torch.cuda.Stream()

    def make():
        ctx = sb.sb_create(n, *q, sb.SB_J_BF16)
        sb.sb_set_factor(ctx, 4, member, couple, 1.0)
        return ctx

    def advance(ctx):
        sb.sb_advance(ctx, variant, 1.0, 0.05, dt, 4, sched, stream=stream)

    ctx, other = make(), make()
    sb.sb_set_option(other, sb.SB_OPT_FACTOR, 0)
    sb.sb_set_state(ctx, x, y)
    if warm:
        advance(ctx)
        sb.sb_set_state(ctx, x, y)
    g = _record(stream, lambda: advance(ctx))
    assert sb.sb_step_kernels(ctx) in ("k_step", "k_step_dsb16")
    qa = inputs.QuboArrays(n, *q)
    for w_c in (None, 1.0, 0.25):
        if w_c:
            for c in (ctx, other):
                _weights(c, qa, w_c)
        sb.sb_set_state(other, x, y)
        advance(other)
        want = sb.sb_get_state(other)
        for _ in range(2):
            sb.sb_set_state(ctx, x, y)
            g.replay()
            got = sb.sb_get_state(ctx)
            assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])


def test_selection_of_the_best_replica_reads_no_caller_memory():
    """best_r and T in one buffer: beyond the four bytes that they share, T is still the
    best replica's."""
    import torch
    q = inputs.random_qubo(300, 9, 5)
    ctx = sb.sb_create(q.n, q.rowptr, q.col, q.val, q.lin)
    sb.sb_run(ctx, "bsb", 1.0, 0.3, 0.4, 20, 8, seed=3)
    T, _, r = sb.sb_best(ctx)
    assert r[0] != 0
    buf = torch.zeros(512, dtype=torch.uint8, device="cuda")
    for _ in range(20):
        buf.zero_()
        sb.sb_readout_device(ctx, None, None, buf[:4].view(torch.int32), buf[:300])
        torch.cuda.synchronize()
        assert np.array_equal(buf[4:300].cpu().numpy(), T[4:])
