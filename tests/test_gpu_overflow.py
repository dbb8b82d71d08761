"""An activation that overflows (float32 sums beyond bfloat16's range) reaches
the outputs whose 27 neighbours include it and no others, also in the training
output layer, whose matrix products pair every staged row with eight output
rows (zero weights where a row is none of theirs)."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _grad(gad, torch, big):
    """Gradient for a field of one positive and one negative point, four rows
    apart in one tile. Channel 0 carries the positive part and channel 1 the
    negative part; layer 3 scales channel 0 by `big`."""
    C, taps = 32, 27
    w = torch.zeros(taps * C + 2 * taps * C * C + taps * C)
    w1 = w[:864].view(taps, C)
    w2 = w[864:864 + 27648].view(taps, C, C)
    w3 = w[864 + 27648:864 + 2 * 27648].view(taps, C, C)
    w4 = w[864 + 2 * 27648:].view(taps, C)
    w1[13, 0], w1[13, 1] = 1.0, -1.0
    w2[13, 0, 0], w2[13, 1, 1] = 1e20, 1.0
    w3[13, 0, 0], w3[13, 1, 1] = big, 1.0
    w4[:, 1] = 0.5
    u = torch.zeros((1, 8, 16, 64))
    u[0, 4, 1, 20], u[0, 4, 5, 20] = 1.0, -1.0
    t = torch.ones_like(u)
    loss, g = gad.guess_grad(w.cuda(), u.cuda(), t.cuda(), 0.1)
    return loss, g.cpu()[864 + 27648:864 + 2 * 27648].view(taps, C, C).numpy()


def test_overflow_stays_with_its_neighbours(gad):
    import torch
    loss0, ok = _grad(gad, torch, 1.0)
    loss1, bad = _grad(gad, torch, 1e20)         # 1e40 in layer 3: inf
    assert np.isfinite(loss0) and not np.isfinite(loss1)
    assert np.isfinite(ok).all() and np.abs(ok[:, :, 1]).max() > 0
    np.testing.assert_array_equal(bad[:, :, 1], ok[:, :, 1])
