"""Factored dSB with FP32 couplings that BF16 does not hold, one to four slots, BF16 and
FP32 U rows: bit-equal to the plain kernel. Couplings are whole numbers of 2^-11 and
a row's sum of them stays below 2^7, so every FP32 sum is exact in any order."""
import numpy as np
import pytest

import paper_2402_14718_gb300 as sb
from tests.test_gpu_factor_blocks import SIZES, _grouped

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R", [8, 64, 256])
@pytest.mark.parametrize("K", [1, 2, 3, 4])
@pytest.mark.parametrize("sizes", [SIZES, SIZES + (300,)])   # 300: FP32 U rows
def test_fp32_heads(R, K, sizes):
    import torch
    w = 1.0 + 2.0 ** -9
    qs, members, couple, off = [], [], None, 0
    for e in range(2):
        (rowptr, col, val, lin), m, couple = _grouped(sizes[e:], K, 200 * K + e)
        qs.append((rowptr, col, np.where(val > 0, val * w, val), lin))
        members.append(np.where(m >= 0, m + off, -1))
        off += len(sizes)
    ctx = sb.sb_create_batch(qs, sb.SB_J_FP32)
    sb.sb_set_factor(ctx, off, np.concatenate(members).astype(np.int32), couple, w)
    assert sb.sb_factor_info(ctx)["rows"] > 0
    rng = np.random.default_rng(R + K)
    x = rng.uniform(-1, 1, size=(ctx.n, R)).astype(np.float32)
    x[rng.random(x.shape) < 0.02] = 0.0
    y = rng.uniform(-0.3, 0.3, size=x.shape).astype(np.float32)
    sched = torch.tensor([0.3, 0.5, 0.7], device="cuda")
    out = []
    for fac, names in ((-1, "k_fac_sum_sgn + k_step_fac_sgn"), (0, "k_step")):
        sb.sb_set_option(ctx, sb.SB_OPT_FACTOR, fac)
        sb.sb_set_state(ctx, x, y)
        sb.sb_advance(ctx, "dsb", 1.0, 0.05, 0.5, 3, sched)
        assert sb.sb_step_kernels(ctx) == names
        out.append(sb.sb_get_state(ctx))
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
