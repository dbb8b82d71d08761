"""The work-list launch of a batched solve on groups too large for one-kernel
solves: 2D and 3D shapes with several element counts and block sizes per
stage, a group whose dot passes end in launches of their own, and a small 2D
group that keeps its one-kernel solve."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _solve(gad, ts, method, lists):
    gad.set_batched_launch(lists)
    try:
        out = gad.deconvolve_batched(ts, [0.1] * len(ts), method=method, tol=0.0, maxit=3)
        return out, gad.last_launch_count()
    finally:
        gad.set_batched_launch(False)


@pytest.mark.parametrize("method", ["vancittert", "cg", "bicgstab", "sd"])
def test_large_groups_equal_branches_and_singles(gad, method):
    import torch
    rng = np.random.default_rng(21)
    shapes = [(1024, 1024)] * 8 + [(384, 384), (288, 512), (64, 64), (48, 64, 32), (72, 48, 96), (384, 384), (64,) * 3]
    ts = [torch.from_numpy(rng.standard_normal(s).astype(np.float32)).cuda() for s in shapes]
    (om, im, sm, hm), launches = _solve(gad, ts, method, True)
    (ob, ib, sb, hb), _ = _solve(gad, ts, method, False)
    assert list(im) == list(ib) == [3] * len(ts) and list(sm) == list(sb)
    for i, t in enumerate(ts):
        np.testing.assert_array_equal(om[i].cpu().numpy(), ob[i].cpu().numpy())
        np.testing.assert_array_equal(hm[i][:4], hb[i][:4])
    for i in (0, 7, 8, 9, 10, 11, 12, 14):
        one = gad.deconvolve(ts[i], 0.1, method=method, tol=0.0, maxit=3, ndim=ts[i].ndim)
        np.testing.assert_array_equal(om[i].cpu().numpy(), one.u.cpu().numpy())
    # with one 1024^2 field instead of eight its dot passes have too few blocks for a launch at their end
    assert launches > _solve(gad, ts[7:], method, True)[1]
