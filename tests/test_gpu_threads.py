"""Two host threads, each with a context of its own, launch the same kernels
with different amounts of shared memory at the same time. A kernel's
shared-memory limit belongs to the process, so a launch must never lower it
under another thread's."""

import ctypes
import threading

import pytest

pytestmark = pytest.mark.gpu


def _spin(lib, gad, torch, nx, batch, dtype, calls, start, out):
    ctx = ctypes.c_void_p()
    assert lib.ad_create(ctypes.byref(ctx), 0) == 0
    g = gad.ad_grid()
    g.ndim, g.dtype, g.gamma = 2, 1 if dtype == torch.float64 else 0, 0.2
    g.n[0], g.n[1] = nx, 8
    u = torch.ones((batch, 8, nx), device="cuda", dtype=dtype)
    v = torch.empty_like(u)
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    start.wait()
    bad = 0
    for _ in range(calls):
        bad += lib.ad_filter(ctx, ctypes.byref(g), u.data_ptr(), v.data_ptr(), batch, s.cuda_stream) != 0
    s.synchronize()
    out[nx] = (bad, float((v - 1.0).abs().max()))
    lib.ad_destroy(ctx)


# inverse x passes of 52,352 and 52,232 bytes (float32), of 78,464 and 52,352 (float64)
@pytest.mark.parametrize("case", [("f32", 3072, 160, 12288, 40), ("f64", 2304, 160, 3072, 80)])
def test_two_threads_with_their_own_contexts(gad, case):
    import torch
    dtype = torch.float64 if case[0] == "f64" else torch.float32
    lib, out, start = gad.load(), {}, threading.Barrier(2)
    ts = [threading.Thread(target=_spin, args=(lib, gad, torch, nx, b, dtype, 2000, start, out))
          for nx, b in (case[1:3], case[3:5])]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert len(out) == 2
    for nx, (bad, err) in out.items():
        assert bad == 0, (nx, bad)
        assert err < 1e-5, (nx, err)            # G keeps a constant field
