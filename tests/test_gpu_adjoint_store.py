"""sd_adjoint keeps every step's positions while they take at most 256 MB and recomputes
segments from checkpoints beyond: a run above the limit against its two halves, each below."""
import numpy as np
import pytest

import paper_1205_6333_gb300 as sd
from paper_1205_6333_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,T,K", [(3000, 3800, 400), (1500, 7600, 1000)])   # (the second: one launch a run of steps)
def test_kept_positions_and_checkpoints_agree(n, T, K):
    assert 24 * n * T > 256 << 20 > 24 * n * (T // 2)
    x0, _ = inputs.cube_rsa(n, 0.02, 601)
    g, dt, half = inputs.normal_forces(n, 602), 1e-4, T // 2
    with sd.System(n, gravity=(0.0, 0.0, -1.0)) as s:
        s.set_positions(x0)
        gx, gF = s.adjoint(dt, T, K, g)                      # checkpoints
        np.testing.assert_array_equal(s.get_positions(), x0)
        s.step(dt, half)
        lam, gF2 = s.adjoint(dt, T - half, K, g)             # kept, a ragged last segment
        s.set_positions(x0)
        gx1, gF1 = s.adjoint(dt, half, K, lam)
        np.testing.assert_array_equal(s.get_positions(), x0)
    np.testing.assert_array_equal(gx1, gx)                   # the same steps, bit for bit
    assert np.abs(gF1 + gF2 - gF).max() <= 1e-12 * np.abs(gF).max()
