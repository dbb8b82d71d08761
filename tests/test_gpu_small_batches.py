"""Batches of small 2D fields on the GPU: a few are solved and filtered by one
thread-block cluster each in a single launch, more than run at once by the
pass kernels. Both against the oracle, with the tolerances of the other GPU
tests (filter 3e-6 and 1e-13, closure and one pass 1e-5 and 1e-12)."""

import numpy as np
import pytest

import oracle
from oracle import closure as oc

pytestmark = pytest.mark.gpu

FEW, MANY = 3, 64                  # 14 clusters of 16 CTAs run at once


def _rel(a, b):
    return np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300)


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("method", ["vancittert", "sd", "cg", "bicgstab"])
def test_solves_of_few_and_many_small_fields(gad, method, dtype):
    import torch
    rng = np.random.default_rng(11)
    shape, tol, prec = ((64, 96), 1e-5, "f32") if dtype == np.float32 else ((128, 64), 1e-12, "f64")
    ub = np.stack([oracle.filter_field(rng.standard_normal(shape), 0.3) for _ in range(MANY)]).astype(dtype)
    ref = [oracle.solve(method, ub[i].astype(np.float64), 0.3, tol=0.0, maxit=1, precision=prec).u for i in (0, 2)]
    for n in (FEW, MANY):
        res = gad.deconvolve(torch.from_numpy(ub[:n]).cuda(), 0.3, method=method, tol=0.0, maxit=1, ndim=2)
        launches = gad.last_launch_count()
        assert launches == 1 if n == FEW else launches > 1, (n, launches)
        assert list(res.iterations) == [1] * n
        for i, r in zip((0, 2), ref):
            assert _rel(res.u[i].double().cpu().numpy(), r) < tol, (n, i)


def test_a_second_round_only_where_it_is_short(gad):
    """20 fields are two rounds of clusters: still one launch on 128^2 float32,
    the pass kernels on 192^2 float32 and 128^2 float64."""
    import torch
    for shape, dtype, one in (((128, 128), torch.float32, True), ((192, 192), torch.float32, False),
                              ((128, 128), torch.float64, False)):
        t = torch.rand((20,) + shape, device="cuda", dtype=dtype)
        gad.deconvolve(t, 0.2, method="cg", tol=0.0, maxit=2, ndim=2)
        assert (gad.last_launch_count() == 1) == one, (shape, dtype)


@pytest.mark.parametrize("dtype,tol", [(np.float32, 3e-6), (np.float64, 1e-13)])
def test_filter_and_closure_of_few_and_many_small_fields(gad, dtype, tol):
    import torch
    rng = np.random.default_rng(12)
    u = rng.standard_normal((MANY, 96, 64)).astype(dtype)
    for n in (FEW, MANY):
        out = gad.filter(torch.from_numpy(u[:n]).cuda(), 0.2, ndim=2).double().cpu().numpy()
        assert (gad.last_launch_count() == 1) == (n == FEW)
        for i in (0, n - 1):
            assert _rel(out[i], oracle.filter_field(u[i].astype(np.float64), 0.2)) < tol, (n, i)
    v = rng.standard_normal((MANY // 2, 2, 48, 64)).astype(dtype)
    for n in (FEW, MANY // 2):
        t = torch.from_numpy(v[:n]).cuda()
        tau = gad.closure(t, t, 0.2, ncomp=2, ndim=2).double().cpu().numpy()
        ref = oc.closure_stress(v[n - 1].astype(np.float64), v[n - 1].astype(np.float64), 0.2)
        assert _rel(tau[n - 1], ref) < (1e-5 if dtype == np.float32 else 1e-12), n
