"""sb_set_weights that runs out of device memory: every kernel of the context runs
with the same couplings afterwards, those with tables of their own included."""
import contextlib
import ctypes

import numpy as np
import pytest

import paper_2402_14718_gb300 as sb

pytestmark = pytest.mark.gpu


@contextlib.contextmanager
def _full(spare_blocks):
    """Device memory taken up in blocks of 2 MiB, `spare_blocks` of them given back."""
    import torch
    rt = ctypes.CDLL("libcudart.so.13")
    rt.cudaFree.argtypes = [ctypes.c_void_p]
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    mb, held = 1 << 20, []
    for size in (1024 * mb, 64 * mb, 2 * mb):
        p = ctypes.c_void_p()
        while rt.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(size)) == 0:
            held.append(p.value)
    rt.cudaGetLastError()
    try:
        for _ in range(spare_blocks):
            rt.cudaFree(held.pop())
        yield
    finally:
        for q in held:
            rt.cudaFree(q)


def test_no_table_keeps_the_old_couplings():
    """A band of 32 couplings a row over 150,000 rows: the tiled kernel's tables, 9.6 MB
    of temporary indices among them, are rebuilt with 8 MiB to spare, and fail."""
    import torch
    n, mb = 150000, 1 << 20
    d = np.concatenate([np.arange(-16, 0), np.arange(1, 17)])
    i = np.arange(n)
    col = np.sort((i[:, None] + d) % n, axis=1).astype(np.int32)
    gap = np.abs(col - i[:, None])
    cls = (np.minimum(gap, n - gap) % 2 == 1).astype(np.int8).ravel()
    val = np.where(cls, 1.0, -1.0)
    ctx = sb.sb_create(n, (32 * np.arange(n + 1)).astype(np.int32), col.ravel(), val,
                       np.full(n, 0.3))
    quality = np.full(n, 0.5)
    sched = torch.linspace(0.2, 0.6, 20, device="cuda")
    rng = np.random.default_rng(4)

    def run(R, steps, key, value):
        x = rng.uniform(-1, 1, size=(n, R)).astype(np.float32)
        out = []
        for v in (-1, value):
            sb.sb_set_option(ctx, key, v)
            sb.sb_set_state(ctx, x, x)
            sb.sb_advance(ctx, "bsb", 1.0, 0.3, 0.4, steps, sched[:steps].contiguous())
            out.append(sb.sb_get_state(ctx)[0])
        sb.sb_set_option(ctx, key, -1)
        return out

    def tables_against_none():
        for R, steps, key in ((1, 20, sb.SB_OPT_R1_LANES), (128, 4, sb.SB_OPT_ROWS_PER_WARP)):
            a, b = run(R, steps, key, 0)
            assert np.array_equal(a, b)

    sb.sb_set_weights(ctx, cls, quality, 1.0, 1.0)
    for _ in range(30):  # enough steps for the one-replica tables
        run(1, 20, sb.SB_OPT_R1_LANES, 0)
    sb.sb_set_option(ctx, sb.SB_OPT_TILED, 1)
    run(32, 2, sb.SB_OPT_ROWS_PER_WARP, -1)
    sb.sb_set_option(ctx, sb.SB_OPT_TILED, 0)
    tables_against_none()
    sigma = sb.sb_info(ctx)["sigma_j"]
    with _full(4), pytest.raises(sb.SbError):
        sb.sb_set_weights(ctx, cls, quality, 1.0, 0.25)
    assert sb.sb_info(ctx)["sigma_j"] < 0.9 * sigma  # the new couplings are in
    tables_against_none()
