"""FP64 readout from selection bits (couplings that are whole numbers of 2^-8)
and through the general FP64 kernel, against the energy of Eq. 13 summed in
numpy, over replica counts at the edges of the kernel's lane teams."""
import numpy as np
import pytest

import paper_2402_14718_gb300 as sb

pytestmark = pytest.mark.gpu


def _qubo(n, seed, weights):
    """Random symmetric QUBO with an empty row, a full row and ragged others."""
    rng = np.random.default_rng(seed)
    B = np.zeros((n, n))
    m = np.triu(rng.random((n, n)) < 6.0 / n, 1)
    m[0, 1:] = True
    m[:, 1] = False
    m[1, :] = False
    B[m] = rng.choice(weights, size=int(m.sum()))
    B = B + B.T
    rowptr = np.concatenate([[0], np.cumsum((B != 0).sum(1))]).astype(np.int32)
    col = np.nonzero(B)[1].astype(np.int32)
    return B, (rowptr, col, B[B != 0], rng.normal(size=n))


@pytest.mark.parametrize("R", [1, 2, 7, 8, 9, 15, 16, 17, 31, 32, 33, 50, 64, 100, 256, 257, 520])
@pytest.mark.parametrize("weights", [(-1.0, 1.0), (-0.75, 2.5, 100.0), (-0.3, 1.0)])
@pytest.mark.parametrize("prec", [sb.SB_J_FP32, sb.SB_J_BF16])
def test_energies_match_the_plain_sum(R, weights, prec):
    import torch
    qs = [_qubo(n, 10 * n + R, weights) for n in (331, 70)]
    ctx = sb.sb_create_batch([q for _, q in qs], prec)
    rng = np.random.default_rng(R)
    x = rng.uniform(-1.0, 1.0, size=(ctx.n, R)).astype(np.float32)
    x[rng.random(x.shape) < 0.05] = 0.0
    T = (x > 0).astype(np.float64)
    ref, r0 = [], 0
    for B, (_, _, _, lin) in qs:
        t = T[r0:r0 + len(lin)]
        ref.append(lin @ t + 0.5 * np.sum(t * (B @ t), axis=0))
        r0 += len(lin)
    ref = np.array(ref)
    # each of at most ~2,600 terms of size <= 100 is rounded at 2^-53 a few times
    tol = dict(rtol=1e-12, atol=1e-12 * max(1.0, np.abs(ref).max()))
    np.testing.assert_allclose(sb.sb_energy(ctx, np.where(T > 0, 1, -1).astype(np.int8)), ref, **tol)
    sb.sb_set_state(ctx, x, np.zeros_like(x))
    np.testing.assert_allclose(sb.sb_energy(ctx, None, R), ref, **tol)
    # device outputs, aligned and not aligned for their type
    for off in (0, 1):
        bE = torch.zeros(2 * R * 8 + 8, dtype=torch.uint8, device="cuda")
        be = torch.zeros(2 * 8 + 8, dtype=torch.uint8, device="cuda")
        br = torch.zeros(2 * 4 + 8, dtype=torch.uint8, device="cuda")
        dT = torch.zeros(ctx.n, dtype=torch.uint8, device="cuda")
        sb.sb_readout_device(ctx, bE.data_ptr() + off, be.data_ptr() + off, br.data_ptr() + off, dT)
        torch.cuda.synchronize()
        E = bE.cpu().numpy()[off:off + 2 * R * 8].view(np.float64).reshape(2, R)
        best = be.cpu().numpy()[off:off + 16].view(np.float64)
        r = br.cpu().numpy()[off:off + 8].view(np.int32)
        np.testing.assert_allclose(E, ref, **tol)
        assert np.array_equal(best, E.min(1)) and np.array_equal(r, E.argmin(1))
        sel = np.concatenate([T[:331, r[0]], T[331:, r[1]]])
        assert np.array_equal(dT.cpu().numpy(), sel.astype(np.uint8))


def test_weights_change_the_form():
    """sb_set_weights to a weight that is no whole number of 2^-8, and back."""
    _, (rowptr, col, val, lin) = _qubo(331, 5, (-1.0, 1.0))
    ctx = sb.sb_create(331, rowptr, col, val, lin)
    cls = (val > 0).astype(np.int8)
    q = np.abs(lin)
    R = 20
    T = np.random.default_rng(1).integers(0, 2, size=(331, R))
    spins = np.where(T > 0, 1, -1).astype(np.int8)
    rows = np.repeat(np.arange(331), np.diff(rowptr))
    for w_c in (1.0, 0.3, 1.0):
        sb.sb_set_weights(ctx, cls, q, 0.7, w_c)
        b = np.where(cls == 0, -1.0, w_c)
        ref = (0.7 * q) @ T + 0.5 * (b[:, None] * T[rows] * T[col]).sum(0)
        np.testing.assert_allclose(sb.sb_energy(ctx, spins)[0], ref, rtol=1e-12, atol=1e-9)
