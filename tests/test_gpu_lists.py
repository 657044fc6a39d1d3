"""The Verlet steps' check and rebuild at the edges of their scan chunks (4,096 buckets) and
force variants, and products at moved positions, against the oracle."""
import numpy as np
import pytest

import oracle
import paper_1205_6333_gb300 as sd
from paper_1205_6333_gb300 import inputs
from helpers import TOL, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rep", [False, True])
@pytest.mark.parametrize("n,prec", [(300, "fp32c"), (2049, "fp64"), (2100, "fp32c"), (4097, "fp32c"), (8193, "fp32c")])
def test_steps_that_rebuild_their_list(n, prec, rep):
    # forces along +-x move neighbours apart by several skins within the run, so the list is
    # rebuilt in most steps
    x0, _ = inputs.cube_rsa(n, 0.05, 501 + n)
    F = np.zeros((n, 3))
    F[:, 0] = np.where(np.arange(n) % 2 == 0, 3.0, -3.0)
    dt, steps = 1.5, 4
    with sd.System(n, prec=prec, dense="symmetric", rep_eps=0.01 if rep else 0.0) as s:
        s.set_positions(x0)
        s.set_forces(F)
        s.step(dt, steps)
        x = s.get_positions()
    ref = oracle.euler(x0, steps, dt, fext=F, rep_eps=0.01 if rep else 0.0, nthreads=16)
    moved = np.abs(ref - x0).max()
    assert moved > 0.25                                  # beyond skin / 2
    assert np.abs(x - ref).max() <= 10 * TOL[prec] * moved


@pytest.mark.parametrize("box", [False, True])
def test_products_and_steps_in_any_order(box):
    # the steps' list and the products' are built when they are first needed
    n = 3000
    x0, L = inputs.cube_rsa(n, 0.05, 511)
    F = inputs.normal_forces(n, 512)
    kw = dict(box=(L, L, L)) if box else {}
    with sd.System(n, prec="fp64", **kw) as s:
        s.set_forces(F)
        for k, x in enumerate((x0, x0 + 0.3 * np.sin(x0))):
            s.set_positions(x)
            v = s.mobility_apply(F)
            gF = s.vjp(F, F)[1]
            if k:
                s.step(0.01, 1)
                x1 = s.get_positions()
                v1 = s.mobility_apply(F)
            ref = oracle.mobility_apply(x, F, "rpy", box=kw.get("box"), nthreads=16)
            assert rel_err(v, ref) <= TOL["fp64"]
            assert rel_err(gF, ref) <= TOL["fp64"]       # mu is symmetric
    assert np.abs(x1 - (x + 0.01 * ref)).max() <= 1e-12 * np.abs(x).max()
    assert rel_err(v1, oracle.mobility_apply(x1, F, "rpy", box=kw.get("box"), nthreads=16)) <= TOL["fp64"]
