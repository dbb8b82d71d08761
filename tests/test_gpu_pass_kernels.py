"""GPU parity of the pass kernels on grids too large for the one-kernel path
of small 2D fields: float64 solves in 2D and 3D, the host-driven loop, fields
that converge at once or are not finite, and lengths with a factor 27.
Tolerances as in test_gpu_solvers.py and test_gpu_filter.py."""

import numpy as np
import pytest

import oracle
from synth import fields
from parity_tools import ensemble_runs, field_tolerance

pytestmark = pytest.mark.gpu

METHODS = ["vancittert", "sd", "cg", "bicgstab"]


def _rel(a, b):
    return np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300)


def _ubar(shape, seed, gamma, dtype):
    if len(shape) == 3:
        u = fields.random_velocity_field(shape, seed, fields.spectrum_3d_kolmogorov)[0]
    else:
        u = fields.random_scalar_field(shape, seed, fields.spectrum_2d_kraichnan)
    return u, oracle.filter_field(u, gamma).astype(dtype)


def _gpu(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("method", METHODS)
@pytest.mark.parametrize("shape", [(192, 192), (96, 256), (48, 36, 24), (16, 24, 64)])
def test_fixed_passes_f64(gad, method, shape):
    _, ub = _ubar(shape, 7, 0.1, np.float64)
    for npass in (1, 3):
        res = gad.deconvolve(_gpu(ub), 0.1, method=method, tol=0.0, maxit=npass, ndim=len(shape))
        assert gad.last_launch_count() > 1
        base, runs = ensemble_runs(method, ub, 0.1, 0.0, npass, "f64")
        tol, spread = field_tolerance(base, runs, "f64")
        err = _rel(res.u.cpu().numpy(), base.u)
        assert err < tol, (npass, err, spread)
        np.testing.assert_allclose(res.history[0, :npass + 1], base.history[:npass + 1], rtol=1e-9)


@pytest.mark.parametrize("method", METHODS)
@pytest.mark.parametrize("shape,dtype", [((192, 192), np.float64), ((48, 36, 24), np.float64)])
def test_initial_guess_one_pass_f64(gad, method, shape, dtype):
    u, ub = _ubar(shape, 8, 0.1, dtype)
    u0 = 0.5 * (ub + u)
    res = gad.deconvolve(_gpu(ub), 0.1, method=method, tol=0.0, maxit=1, u0=_gpu(u0), ndim=len(shape),
                         true_residual=True)
    ref = oracle.solve(method, ub, 0.1, tol=0.0, maxit=1, u0=u0)
    assert _rel(res.u.cpu().numpy(), ref.u) < 1e-12
    np.testing.assert_allclose(res.history[0], ref.history, rtol=1e-11)
    np.testing.assert_allclose(res.true_residual[0], res.history[0, 1], rtol=1e-6)


@pytest.mark.parametrize("shape,dtype", [((512, 512), np.float32), ((192, 192), np.float64), ((48, 36, 24), np.float32)])
def test_graph_and_host_loop_agree(gad, shape, dtype):
    _, ub = _ubar(shape, 6, 0.1, dtype)
    t = _gpu(ub)
    for method in METHODS:
        runs = []
        for graph in (True, False):
            gad.set_graph_mode(graph)
            try:
                r = gad.deconvolve(t, 0.1, method=method, tol=1e-4, maxit=300, ndim=len(shape))
                assert gad.last_launch_count() > 1
                runs.append(r)
            finally:
                gad.set_graph_mode(True)
        a, b = runs
        assert int(a.iterations[0]) == int(b.iterations[0]) > 0 and a.status[0] == b.status[0]
        np.testing.assert_array_equal(a.u.cpu().numpy(), b.u.cpu().numpy())
        n = int(a.iterations[0]) + 1
        np.testing.assert_array_equal(a.history[0, :n], b.history[0, :n])


@pytest.mark.parametrize("shape,dtype", [((288, 256), np.float32), ((144, 128), np.float64), ((24, 32, 48), np.float32)])
def test_edge_cases_per_field_status(gad, shape, dtype):
    """A regular field, a zero field, a constant field and a field holding a NaN
    in one batch: per-field statuses, the regular field's result bitwise that of
    its solve alone and repeatable; no pass at all with maxit = 0."""
    _, ub = _ubar(shape, 2, 0.1, dtype)
    batch = np.stack([ub, np.zeros_like(ub), np.full_like(ub, 2.5), ub.copy()])
    batch[(3,) + (5,) * len(shape)] = np.nan
    nd = len(shape)
    for method in METHODS:
        res, again = (gad.deconvolve(_gpu(batch), 0.1, method=method, tol=1e-4, maxit=2000, ndim=nd) for _ in range(2))
        alone = gad.deconvolve(_gpu(ub), 0.1, method=method, tol=1e-4, maxit=2000, ndim=nd)
        assert int(res.status[0]) == gad.AD_OK and res.iterations[0] == alone.iterations[0]
        np.testing.assert_array_equal(res.u[0].cpu().numpy(), alone.u.cpu().numpy())
        np.testing.assert_array_equal(res.u[:3].cpu().numpy(), again.u[:3].cpu().numpy())
        assert int(res.status[1]) == gad.AD_OK and int(res.iterations[1]) == 0
        assert int(res.status[2]) == gad.AD_OK and int(res.iterations[2]) == 0
        assert int(res.status[3]) == gad.AD_ERR_NONFINITE
        np.testing.assert_array_equal(res.u[1].cpu().numpy(), 0.0)
        np.testing.assert_array_equal(res.u[2].cpu().numpy(), 2.5)
        none = gad.deconvolve(_gpu(ub), 0.1, method=method, tol=1e-6, maxit=0, ndim=nd)
        assert int(none.status[0]) == gad.AD_MAXIT and int(none.iterations[0]) == 0
        np.testing.assert_array_equal(none.u.cpu().numpy(), ub)


def test_single_mode_terminates_in_one_pass(gad):
    n = 256
    x = 2 * np.pi * np.arange(n) / n
    X, Y = np.meshgrid(x, x)
    u = np.cos(3 * X + 5 * Y)
    ub = oracle.filter_field(u, 0.2)
    for method in ("sd", "cg", "bicgstab"):
        res = gad.deconvolve(_gpu(ub), 0.2, method=method, tol=1e-10, maxit=10)
        assert gad.last_launch_count() > 1
        assert int(res.iterations[0]) == 1 and int(res.status[0]) == gad.AD_OK, method
        np.testing.assert_allclose(res.u.cpu().numpy(), u, atol=1e-12)


# float32 lengths with a factor 27 or 81, which have plans of fused radices and no kernel of their own; 1296 on
# the last axis and 972 in x (rows of 486) have had a plan since those radices only
@pytest.mark.parametrize("shape", [(108, 512), (216, 384), (432, 288), (864, 128), (972, 64), (1296, 64), (1728, 32),
                                   (256, 216), (256, 432), (64, 864), (64, 972), (64, 1296), (32, 108, 64),
                                   (32, 216, 32), (54, 54, 108)])
def test_lengths_with_a_factor_27(gad, shape):
    import torch
    rng = np.random.default_rng(sum(shape))
    u = rng.standard_normal((2,) + shape).astype(np.float32)
    out = gad.filter(torch.from_numpy(u).cuda(), 0.2, ndim=len(shape)).double().cpu().numpy()
    for b in range(2):
        assert _rel(out[b], oracle.filter_field(u[b].astype(np.float64), 0.2)) < 3e-6
    ub = oracle.filter_field(u[0].astype(np.float64), 0.2).astype(np.float32)
    for method in ("cg", "bicgstab"):
        res = gad.deconvolve(_gpu(ub), 0.2, method=method, tol=0.0, maxit=1, ndim=len(shape))
        ref = oracle.solve(method, ub.astype(np.float64), 0.2, tol=0.0, maxit=1, precision="f32")
        assert _rel(res.u.double().cpu().numpy(), ref.u) < 1e-5, method


def test_batched_with_autotune_above_the_one_kernel_grids(gad):
    data = []
    for i, shape in enumerate([(288, 384), (576, 192), (384, 288), (36, 48, 48)]):
        data.append(_ubar(shape, 20 + i, 0.1, np.float32)[1])
    ts = [_gpu(a) for a in data]
    singles = [gad.deconvolve(t, 0.1, method="cg", tol=1e-4, maxit=800, ndim=t.ndim) for t in ts]
    gad.autotune(for_batched=True)
    try:
        outs, its, sts, _ = gad.deconvolve_batched(ts, [0.1] * len(ts), method="cg", tol=1e-4, maxit=800)
    finally:
        gad.autotune(for_batched=False)
    for i, single in enumerate(singles):
        assert sts[i] == gad.AD_OK and abs(int(its[i]) - int(single.iterations[0])) <= 2
        # both residuals are within tol; iterates that stop a pass apart differ by about the step
        assert _rel(outs[i].cpu().numpy(), single.u.cpu().numpy()) < 1e-3
