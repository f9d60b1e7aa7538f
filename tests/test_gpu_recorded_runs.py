"""Runs and readouts that a caller recorded into a CUDA graph, replayed after
sb_set_weights gave the context new couplings: they read the context's
couplings in place, so a replay gives what a fresh call gives."""
import numpy as np
import pytest

import paper_2402_14718_gb300 as sb
from tests import inputs

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
