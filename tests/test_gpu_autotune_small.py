"""The tuner on grids that a method solves in one kernel: it leaves the tiles of
the plan's other solves alone."""

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


# shapes used by no other test: plans stay in the context
@pytest.mark.parametrize("shape", [(96, 216), (216, 72), (108, 144), (72, 288)])
def test_tuning_a_one_kernel_method_changes_nothing(gad, shape):
    import torch
    rng = np.random.default_rng(31)
    t = torch.from_numpy(oracle.filter_field(rng.standard_normal(shape), 0.2).astype(np.float32)).cuda()
    before = {m: gad.deconvolve(t, 0.2, method=m, tol=0.0, maxit=4) for m in ("cg", "pcg")}
    gad.autotune(shape, 0.2, batch=1, method="cg")
    for m, b in before.items():
        a = gad.deconvolve(t, 0.2, method=m, tol=0.0, maxit=4)
        np.testing.assert_array_equal(a.u.cpu().numpy(), b.u.cpu().numpy())
        np.testing.assert_array_equal(a.history, b.history)
