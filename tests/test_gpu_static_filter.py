"""ad_filter_static runs the passes that ad_filter launches, in the same tiles.
Its twiddle factors come from the device's float64 sine and cosine, the
context's from the host's long double: in float32 both round to the same
values but for a rare tie, and the results agree to less than one ulp; in
float64 they differ by an ulp or two, and both are compared with the oracle."""

import ctypes

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


# forward and inverse x passes with tiles of their own; ragged; a batch that changes the tiles; 2D and 3D
@pytest.mark.parametrize("shape,batch", [((1024, 512), 1), ((96, 72, 144), 1), ((64, 64, 64), 4), ((48, 24, 36), 3),
                                         ((512, 768), 2), ((16, 8, 12), 1)])
@pytest.mark.parametrize("dtype,tol", [("f32", 3e-6), ("f64", 1e-13)])
def test_static_filter_in_the_same_tiles(gad, shape, batch, dtype, tol):
    import torch
    lib = gad.load()
    lib.ad_filter_static.argtypes = [ctypes.POINTER(gad.ad_grid), ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int,
                                     ctypes.c_void_p]
    lib.ad_filter_static.restype = ctypes.c_int
    g = gad.ad_grid()
    g.ndim, g.dtype, g.gamma = len(shape), gad.AD_F32 if dtype == "f32" else gad.AD_F64, 0.2
    for i, n in enumerate(reversed(shape)):
        g.n[i] = n
    rng = np.random.default_rng(41)
    u = torch.tensor(rng.standard_normal((batch,) + shape), device="cuda",
                     dtype=torch.float32 if dtype == "f32" else torch.float64)
    out = torch.full_like(u, float("nan"))
    assert lib.ad_filter_static(ctypes.byref(g), u.data_ptr(), out.data_ptr(), batch,
                                torch.cuda.current_stream().cuda_stream) == gad.AD_OK
    ref = gad.filter(u, 0.2, ndim=len(shape)).double().cpu().numpy()
    got = out.double().cpu().numpy()
    for b in range(batch):
        ora = oracle.filter_field(u[b].double().cpu().numpy(), 0.2)
        assert np.linalg.norm(got[b] - ora) / np.linalg.norm(ora) < tol
        assert np.linalg.norm(ref[b] - ora) / np.linalg.norm(ora) < tol
        if dtype == "f32":
            assert np.linalg.norm(got[b] - ref[b]) / np.linalg.norm(ref[b]) < 2.0 ** -23
