"""GPU parity of the kernels that a grid's size selects: solves of small 2D
grids by one thread-block cluster, the pass kernels compiled for lengths with
a factor 3, dot passes of many blocks finished by a launch of their own, and
the network layers on rows and planes that do not fill their tiles.

Tolerances are those of the other GPU tests: the filter 3e-6 (float32) and
1e-13 (float64), one pass 1e-5 and 1e-12, the network 3e-2 (bf16 activations,
2^-8 per layer) and gradients with cosine > 0.98."""

import numpy as np
import pytest

import oracle
from oracle import cnn
from synth import fields

pytestmark = pytest.mark.gpu


def _rel(a, b):
    return np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300)


# (Ny, Nx): one CTA; a side with a factor 3; short and long rows; 16 CTAs with a
# partly filled last one; the largest float32 grid
@pytest.mark.parametrize("shape", [(8, 12), (12, 36), (36, 24), (1024, 64), (64, 1024), (144, 96), (256, 256)])
@pytest.mark.parametrize("method", ["vancittert", "sd", "cg", "bicgstab"])
def test_cluster_solve_one_pass(gad, shape, method):
    import torch
    rng = np.random.default_rng(sum(shape))
    for dtype, tol in ((np.float32, 1e-5), (np.float64, 1e-12)):
        if dtype == np.float64 and shape[0] * shape[1] > 128 * 128:
            continue
        ub = oracle.filter_field(rng.standard_normal(shape), 0.3).astype(dtype)
        u0 = (ub + 0.1 * rng.standard_normal(shape)).astype(dtype)
        prec = "f32" if dtype == np.float32 else "f64"
        for guess in (None, u0):
            t = None if guess is None else torch.from_numpy(guess).cuda()
            res = gad.deconvolve(torch.from_numpy(ub).cuda(), 0.3, method=method, tol=0.0, maxit=1, u0=t,
                                 true_residual=True)
            ref = oracle.solve(method, ub.astype(np.float64), 0.3, tol=0.0, maxit=1, precision=prec,
                               u0=None if guess is None else guess.astype(np.float64))
            assert int(res.iterations[0]) == 1 and int(res.status[0]) == gad.AD_MAXIT
            assert _rel(res.u.double().cpu().numpy(), ref.u) < tol, (dtype, guess is None)
            np.testing.assert_allclose(res.history[0], ref.history, rtol=10 * tol)
            np.testing.assert_allclose(res.true_residual[0], res.history[0, 1], rtol=1e-3)


def test_cluster_closure(gad):
    """The closure stress of a small grid (products and stress fused into the
    cluster's prologue and epilogue) against the oracle."""
    import torch
    from oracle import closure as oc
    rng = np.random.default_rng(5)
    v = rng.standard_normal((2, 2, 48, 64))
    w = rng.standard_normal((2, 2, 48, 64))
    tau = gad.closure(torch.from_numpy(v).cuda(), torch.from_numpy(w).cuda(), 0.2, ncomp=2, ndim=2).cpu().numpy()
    for i in range(2):
        assert _rel(tau[i], oc.closure_stress(v[i], w[i], 0.2)) < 1e-13


# every length with kernels of its own, on each axis it serves: rows (Nx = 2L), the last axis, and y in 3D
@pytest.mark.parametrize("n", [36, 48, 72, 96, 144, 192, 288, 384, 576, 768, 1152, 1536, 2304])
def test_filter_lengths_with_a_factor_3(gad, n):
    import torch
    rng = np.random.default_rng(n)
    shapes = [(n, 512)] + ([(256, 2 * n)] if n <= 768 else []) + ([(32, n, 64)] if n <= 576 else [])
    for shape in shapes:
        u = rng.standard_normal((2,) + shape).astype(np.float32)
        out = gad.filter(torch.from_numpy(u).cuda(), 0.2, ndim=len(shape)).double().cpu().numpy()
        for b in range(2):
            assert _rel(out[b], oracle.filter_field(u[b].astype(np.float64), 0.2)) < 3e-6, shape


@pytest.mark.parametrize("space", ["physical", "spectral"])
@pytest.mark.parametrize("method", ["cg", "bicgstab"])
def test_finish_launch_equals_ticket(gad, method, space):
    """Eight 1024^2 fields (thousands of blocks per dot pass, finished by a
    launch of their own) bitwise equal to the same fields solved one by one
    (hundreds of blocks, finished by the last of them)."""
    import torch
    rng = np.random.default_rng(7)
    ub = torch.from_numpy(rng.standard_normal((8, 1024, 1024)).astype(np.float32)).cuda()
    res = gad.deconvolve(ub, 0.1, method=method, tol=0.0, maxit=3, ndim=2, space=space)
    for b in (0, 7):
        alone = gad.deconvolve(ub[b].contiguous(), 0.1, method=method, tol=0.0, maxit=3, space=space)
        np.testing.assert_array_equal(res.u[b].cpu().numpy(), alone.u.cpu().numpy())
        np.testing.assert_array_equal(res.history[b], alone.history[0])


def _to_lib(ws):
    return np.concatenate([np.transpose(ws[0][:, 0], (1, 2, 3, 0)).ravel(),
                           np.transpose(ws[1], (2, 3, 4, 1, 0)).ravel(),
                           np.transpose(ws[2], (2, 3, 4, 1, 0)).ravel(),
                           np.transpose(ws[3][0], (1, 2, 3, 0)).ravel()]).astype(np.float32)


# rows not a multiple of the tiles' 4 and 8; one and two x segments; the tcgen05 layers' uneven shares
@pytest.mark.parametrize("shape", [(8, 18, 64), (12, 18, 32), (12, 18, 128)])
def test_network_on_ragged_rows(gad, shape):
    import torch
    gamma, n = 0.1, 2
    ws = cnn.init_weights(channels=32, seed=6, scale_last=1.0)
    ws[3] *= 0.05
    w = torch.from_numpy(_to_lib(ws)).cuda()
    rng = np.random.default_rng(sum(shape))
    ut = rng.standard_normal((n,) + shape)
    ub = np.stack([oracle.filter_field(u, gamma) for u in ut]).astype(np.float32)
    u0 = gad.guess_infer(w, torch.from_numpy(ub).cuda(), gamma).double().cpu().numpy()
    loss, grad = gad.guess_grad(w, torch.from_numpy(ub).cuda(), torch.from_numpy(ut.astype(np.float32)).cuda(), gamma)
    A, ref_loss, ref = cnn.output_scale(gamma), 0.0, [np.zeros_like(x) for x in ws]
    for b in range(n):
        x = ub[b].astype(np.float64)
        out, _ = cnn.forward(ws, x, A)
        assert _rel(u0[b] - x, out - x) < 3e-2
        L, gs = cnn.loss_and_grads(ws, x, ut[b].astype(np.float32).astype(np.float64), A)
        ref_loss += L / n
        ref = [r + g / n for r, g in zip(ref, gs)]
    assert abs(loss - ref_loss) < 2e-2 * ref_loss
    a, r = grad.double().cpu().numpy(), _to_lib(ref).astype(np.float64)
    cut = np.cumsum([0, 864, 27648, 27648, 864])
    for i in range(4):
        x, y = a[cut[i]:cut[i + 1]], r[cut[i]:cut[i + 1]]
        assert float(np.dot(x, y) / (np.linalg.norm(x) * np.linalg.norm(y))) > 0.98, i
