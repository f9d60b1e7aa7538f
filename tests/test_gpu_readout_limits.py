"""Readout where device memory is short: the selection bits are a faster way to the
energies, and a readout that has no room for them takes the FP64 sums."""
import numpy as np
import pytest

import paper_2402_14718_gb300 as sb
from tests.test_gpu_new_weights import _full
from tests.test_gpu_recorded_runs import _ring

pytestmark = pytest.mark.gpu


def test_no_room_for_the_bits():
    """200,000 rows at 512 replicas: 18.3 MiB of bits and their block sums (22 in whole
    blocks of 2) or 12.2 MiB of FP64 block sums (14), with 18 MiB left over."""
    n, R = 200000, 512
    q = _ring(n)
    x = np.random.default_rng(3).uniform(-1, 1, size=(n, R)).astype(np.float32)

    def energies(spare):
        ctx = sb.sb_create(q.n, q.rowptr, q.col, q.val, q.lin)
        sb.sb_set_state(ctx, x, x)
        if spare is None:
            return sb.sb_energy(ctx, None, R)
        with _full(spare):
            return [sb.sb_energy(ctx, None, R) for _ in range(2)]

    want = energies(None)
    for got in energies(9):
        assert np.allclose(got, want, rtol=1e-12, atol=0)
