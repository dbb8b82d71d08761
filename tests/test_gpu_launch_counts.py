"""Launches reported for a timed pass: one with dots of many blocks is two, the
pass and the launch that finishes its sums."""

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,per", [(8, 2), (1, 1)])
def test_time_pass_counts_the_finish_launch(gad, batch, per):
    reps = 4
    passes = gad.time_passes((1024, 1024), 0.1, batch, method="bicgstab", reps=reps)
    assert passes[-1]["kind"] == "xinv" or "inv" in passes[-1]["kind"]
    assert gad.last_launch_count() == (reps + 1) * per          # of the last pass, which has two dots
