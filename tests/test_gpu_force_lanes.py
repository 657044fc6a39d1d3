"""The two forms of the list's force kernel on either side of the line between them: one step each
against a step without list reuse."""
import numpy as np
import pytest

import paper_1205_6333_gb300 as sd
from paper_1205_6333_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [10751, 10752])
@pytest.mark.parametrize("lub", [False, True])
def test_forces_either_side_of_the_line(n, lub):
    m = 23
    x = 2.3 * np.stack(np.meshgrid(*[np.arange(m)] * 3, indexing="ij"), -1).reshape(-1, 3)[:n]
    x = x + np.random.default_rng(921).uniform(-0.1, 0.1, x.shape)
    F = inputs.normal_forces(n, 922)
    kw = dict(prec="fp64", lubrication=lub, rep_eps=0.0 if lub else 1.0, r_near=2.5)
    out = []
    for skin in (None, -1.0):
        with sd.System(n, verlet_skin=skin, **kw) as s:
            s.set_positions(x)
            s.set_forces(F)
            s.step(1e-3, 2)
            out.append(s.get_positions())
    moved = np.abs(out[1] - x).max()
    assert moved > 1e-4 and np.abs(out[0] - out[1]).max() <= 1e-12 * np.abs(x).max()   # sums in another order
