"""Steps with forces that follow the positions, on a system so crowded that the near-pair list is full:
the particles it leaves out are corrected with this step's forces, not the last one's."""
import numpy as np
import pytest

import oracle
import paper_1205_6333_gb300 as sd
from paper_1205_6333_gb300 import inputs
from helpers import TOL

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp32c", "fp64"])
@pytest.mark.parametrize("skin", [None, -1.0])
def test_crowded_steps_with_repulsion_match_oracle(prec, skin):
    m, eps, dt, steps = 11, 1e-5, 0.02, 3
    rng = np.random.default_rng(911)
    x = 0.9 * np.stack(np.meshgrid(*[np.arange(m)] * 3, indexing="ij"), -1).reshape(-1, 3)
    x = x + rng.uniform(-0.04, 0.04, x.shape)               # some 100 partners within r_near + skin, 32 listed
    n = x.shape[0]
    F = inputs.normal_forces(n, 912)
    ref = oracle.euler(x, steps, dt, fext=F, rep_eps=eps, nthreads=16)
    rep_only = oracle.euler(x, 1, dt, fext=F, rep_eps=eps, nthreads=16) - oracle.euler(x, 1, dt, fext=F, nthreads=16)
    moved = np.abs(ref - x).max()
    assert np.abs(rep_only).max() > 0.01 * moved              # the repulsion matters
    with sd.System(n, prec=prec, rep_eps=eps, verlet_skin=skin) as s:
        s.set_positions(x)
        s.set_forces(F)
        s.step(dt, steps)
        assert np.abs(s.get_positions() - ref).max() <= 10 * TOL[prec] * moved
