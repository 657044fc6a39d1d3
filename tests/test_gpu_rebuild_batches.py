"""The gated rebuild of the steps' list (one cluster, four particles or buckets a thread at a time) at
sizes around its batches, buckets of one, two and many particles, rebuilt in every step: against
the same steps without list reuse."""
import numpy as np
import pytest

import paper_1205_6333_gb300 as sd
from paper_1205_6333_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,crowd,rep,box", [(2047, 0, 0.01, False), (2049, 40, 0.0, False), (8191, 40, 0.0, True),
                                             (8193, 0, 0.01, True), (16385, 300, 0.0, False), (20001, 0, 0.01, False)])
def test_rebuild_in_every_step(n, crowd, rep, box):
    x, L = inputs.cube_rsa(n, 0.05, 901)
    rng = np.random.default_rng(902)
    if crowd:
        x[rng.choice(n, crowd, replace=False)] = x[0] + rng.uniform(-2.0, 2.0, (crowd, 3))
    F = inputs.normal_forces(n, 903)
    F /= np.linalg.norm(F, axis=1)[:, None]
    kw = dict(prec="fp64", rep_eps=rep, dense="symmetric", box=(L + 3.0,) * 3 if box else None)
    out = []
    for skin in (None, -1.0):
        with sd.System(n, verlet_skin=skin, **kw) as s:
            s.set_positions(x)
            s.set_forces(F)
            v = s.mobility_apply(F)
            dt = 0.3 / np.linalg.norm(v - v[0], axis=1).max()      # beyond skin / 4 in every step
            for k in range(6):
                s.step(dt if k % 2 == 0 else -0.9 * dt, 1)
            out.append(s.get_positions())
    moved = np.abs(out[1] - x).max()
    assert moved > 0.02
    assert np.abs(out[0] - out[1]).max() <= 1e-11 * max(1.0, moved)   # rounding of the sums' order, six steps
