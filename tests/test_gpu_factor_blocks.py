"""Group sums and row step of the factored dSB product over block sizes on both
sides of a lane group's and a CTA's share (1 .. 200 members), one to four
slots, every lane-group width, BF16 and FP32 U rows, one and several events:
bit-equal to the plain kernel (all sums are exact)."""
import numpy as np
import pytest

import paper_2402_14718_gb300 as sb

pytestmark = pytest.mark.gpu


def _grouped(sizes, K, seed):
    """QUBO of groups of the given sizes (all members in random slots, unit weight
    between coupled slots) with random +-1 pairs on top."""
    rng = np.random.default_rng(seed)
    n = sum(sizes)
    couple = np.eye(K, dtype=np.uint8)
    for s in range(K - 1):
        couple[s, s + 1] = couple[s + 1, s] = 1
    perm = rng.permutation(n)
    member = np.full((n, K), -1, np.int32)
    B = np.zeros((n, n))
    at = 0
    for g, m in enumerate(sizes):
        rows = perm[at:at + m]
        at += m
        slot = rng.integers(0, K, size=m)
        member[rows, slot] = g
        B[np.ix_(rows, rows)] += couple[np.ix_(slot, slot)]
    extra = np.triu(rng.random((n, n)) < 3.0 / n, 1)
    B += np.where(extra | extra.T, -1.0, 0.0)
    np.fill_diagonal(B, 0.0)
    rowptr = np.concatenate([[0], np.cumsum((B != 0).sum(1))]).astype(np.int32)
    return (rowptr, np.nonzero(B)[1].astype(np.int32), B[B != 0], rng.uniform(0, 1, n)), member, couple


SIZES = (1, 2, 3, 4, 5, 8, 9, 16, 31, 32, 33, 34, 40, 63, 64, 65, 130, 200)


@pytest.mark.parametrize("R", [8, 16, 32, 50, 64, 128, 256, 512])
@pytest.mark.parametrize("K", [1, 2, 3, 4])
@pytest.mark.parametrize("sizes", [SIZES, SIZES + (300,)])   # 300: FP32 U rows
def test_dsb_blocks_bit_for_bit(R, K, sizes):
    import torch
    prec = sb.SB_J_BF16 if R % 3 else sb.SB_J_FP32
    qs, members, couple, off = [], [], None, 0
    for e in range(2):
        q, m, couple = _grouped(sizes[e:], K, 100 * K + e)
        qs.append(q)
        members.append(np.where(m >= 0, m + off, -1))
        off += len(sizes)
    ctx = sb.sb_create_batch(qs, prec)
    sb.sb_set_factor(ctx, off, np.concatenate(members).astype(np.int32), couple, 1.0)
    info = sb.sb_factor_info(ctx)
    assert info["rows"] > 0
    rng = np.random.default_rng(R)
    x = rng.uniform(-1, 1, size=(ctx.n, R)).astype(np.float32)
    x[rng.random(x.shape) < 0.02] = 0.0
    y = rng.uniform(-0.3, 0.3, size=x.shape).astype(np.float32)
    sched = torch.tensor([0.3, 0.5, 0.7], device="cuda")
    out = []
    for fac in (-1, 0):
        sb.sb_set_option(ctx, sb.SB_OPT_FACTOR, fac)
        sb.sb_set_state(ctx, x, y)
        sb.sb_advance(ctx, "dsb", 1.0, 0.05, 0.5, 3, sched)
        out.append(sb.sb_get_state(ctx))
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
