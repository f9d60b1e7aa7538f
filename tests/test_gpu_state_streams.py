"""States passed in and out of device memory beside a stream that does not wait for
the default stream: sb_set_state and sb_get_state have finished when they
return, so the next call on any stream sees the whole state."""
import numpy as np
import pytest

import paper_2402_14718_gb300 as sb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R", [50, 64, 99])
def test_set_advance_get_on_a_side_stream(R):
    """A ring of 400,000 rows: copying the state takes longer than starting a step."""
    import torch
    n = 400000
    i = np.arange(n)
    col = np.sort((i[:, None] + np.array([-7, -1, 1, 7])) % n, axis=1).ravel().astype(np.int32)
    ctx = sb.sb_create(n, (4 * np.arange(n + 1)).astype(np.int32), col, np.ones(4 * n),
                       np.full(n, 0.3))
    g = torch.Generator(device="cuda").manual_seed(R)
    x = 2 * torch.rand((n, R), generator=g, device="cuda") - 1
    y = 0.6 * torch.rand((n, R), generator=g, device="cuda") - 0.3
    sched = torch.linspace(0.2, 0.6, 2, device="cuda")
    side = torch.cuda.Stream()
    out = [torch.empty_like(x) for _ in range(4)]

    def get(a, b):
        sb._lib.check(sb.lib.sb_get_state(ctx.handle, a.data_ptr(), b.data_ptr(), 1))

    def two_runs(wait):
        res = []
        sb.sb_set_state(ctx, x, y)
        for k in (0, 2):
            wait()
            sb.sb_advance(ctx, "bsb", 1.0, 0.3, 0.4, 2, sched, stream=side)
            wait()
            get(out[k], out[k + 1])
            wait()
            with torch.cuda.stream(side):  # reads the copy, then the next run overwrites the state
                res += [out[k].clone(), out[k + 1].clone()]
        torch.cuda.synchronize()
        return res

    want = two_runs(torch.cuda.synchronize)
    assert not torch.equal(want[0], want[2])
    for _ in range(5):
        got = two_runs(lambda: None)
        assert all(torch.equal(a, b) for a, b in zip(got, want))


@pytest.mark.parametrize("n", [1, 7, 300, 40000])
@pytest.mark.parametrize("R", [2, 3, 31, 33, 50, 64, 130])
def test_both_arrays_or_one(n, R):
    """Rows shorter and longer than a warp, x and y together and each alone."""
    import torch
    ctx = sb.sb_create(n, np.zeros(n + 1, np.int32), np.zeros(0, np.int32), np.zeros(0), np.zeros(n))
    g = torch.Generator(device="cuda").manual_seed(n + R)
    x, y = (torch.rand((n, R), generator=g, device="cuda") for _ in range(2))
    sb.sb_set_state(ctx, x, y)
    hx, hy = sb.sb_get_state(ctx)
    assert np.array_equal(hx, x.cpu().numpy()) and np.array_equal(hy, y.cpu().numpy())
    for want_x, want_y in ((1, 1), (1, 0), (0, 1)):
        a, b = torch.full_like(x, 7.0), torch.full_like(y, 7.0)
        sb._lib.check(sb.lib.sb_get_state(ctx.handle, a.data_ptr() if want_x else None,
                                          b.data_ptr() if want_y else None, 1))
        assert torch.equal(a, x) if want_x else bool((a == 7.0).all())
        assert torch.equal(b, y) if want_y else bool((b == 7.0).all())


@pytest.mark.parametrize("R", [50, 64])
def test_get_state_from_several_threads(R):
    """sb_get_state reads a context that it does not change: threads may call it at once."""
    from concurrent.futures import ThreadPoolExecutor
    n = 30000
    ctx = sb.sb_create(n, np.zeros(n + 1, np.int32), np.zeros(0, np.int32), np.zeros(0), np.zeros(n))
    rng = np.random.default_rng(R)
    x, y = (rng.random((n, R), dtype=np.float32) for _ in range(2))
    sb.sb_set_state(ctx, x, y)

    def get(k):
        out = np.zeros((n, R), np.float32)
        p = out.ctypes.data
        sb._lib.check(sb.lib.sb_get_state(ctx.handle, p if k % 2 else None, None if k % 2 else p, 0))
        return np.array_equal(out, x if k % 2 else y)

    with ThreadPoolExecutor(8) as ex:
        assert all(ex.map(get, range(160)))


@pytest.mark.parametrize("pieces", [False, True])
def test_buffers_that_end_with_their_memory(pieces):
    """A kernel is given a buffer only when all of it is allocated: ones that fill their
    allocation to the last byte, and ones that torch maps in several pieces, count."""
    import torch
    n, R = 65536, 50  # 12.5 MiB: exactly 6.25 pieces of 2 MiB
    code = f"""if True:
        import ctypes, torch
        import paper_2402_14718_gb300 as sb
        import numpy as np
        rt = ctypes.CDLL("libcudart.so.13")
        rt.cudaMemcpy.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_size_t, ctypes.c_int]
        n, R, pieces = {n}, {R}, {pieces}
        ctx = sb.sb_create(n, np.zeros(n + 1, np.int32), np.zeros(0, np.int32), np.zeros(0), np.zeros(n))
        x = torch.rand((n, R), device="cuda")
        y = x + 1
        if pieces:
            a, b = torch.zeros_like(x), torch.zeros_like(x)
            pa, pb = a.data_ptr(), b.data_ptr()
        else:
            pa, pb = ctypes.c_void_p(), ctypes.c_void_p()
            assert rt.cudaMalloc(ctypes.byref(pa), ctypes.c_size_t(n * R * 4)) == 0
            assert rt.cudaMalloc(ctypes.byref(pb), ctypes.c_size_t(n * R * 4)) == 0
            a, b = torch.zeros_like(x), torch.zeros_like(x)
        sb.sb_set_state(ctx, x, y)
        sb._lib.check(sb.lib.sb_get_state(ctx.handle, pa, pb, 1))
        if not pieces:
            rt.cudaMemcpy(a.data_ptr(), pa, n * R * 4, 3)
            rt.cudaMemcpy(b.data_ptr(), pb, n * R * 4, 3)
        assert torch.equal(a, x) and torch.equal(b, y)
    """
    import os
    import subprocess
    import sys
    env = dict(os.environ)
    if pieces:
        env["PYTORCH_CUDA_ALLOC_CONF"] = "expandable_segments:True"
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", code], cwd=root, env=env, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]


@pytest.mark.parametrize("R", [1, 50, 64])
@pytest.mark.parametrize("shift", [1, 2, 4])
def test_buffers_off_the_16_byte_boundary(R, shift):
    import torch
    n = 5000
    ctx = sb.sb_create(n, np.zeros(n + 1, np.int32), np.zeros(0, np.int32), np.zeros(0), np.zeros(n))
    g = torch.Generator(device="cuda").manual_seed(R)
    base = torch.rand(2 * n * R + 16, generator=g, device="cuda")
    x, y = base[shift:shift + n * R].view(n, R), base[n * R + 8:2 * n * R + 8].view(n, R)
    sb.sb_set_state(ctx, x, y)
    out = torch.zeros(2 * n * R + 16, device="cuda")
    a, b = out[shift:shift + n * R].view(n, R), out[n * R + 8:2 * n * R + 8].view(n, R)
    sb._lib.check(sb.lib.sb_get_state(ctx.handle, a.data_ptr(), b.data_ptr(), 1))
    assert torch.equal(a, x) and torch.equal(b, y)
    assert out[:shift].sum() == 0 and out[2 * n * R + 8:].sum() == 0
