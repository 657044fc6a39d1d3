"""The steps' list is built when it is first needed, at positions that other calls may have
moved since they were set (a small system's steps, sharded steps): the candidates have to be
screened at those positions, or pairs that came close in between are left out."""
import numpy as np
import pytest

import oracle
import paper_1205_6333_gb300 as sd
from paper_1205_6333_gb300 import inputs
from helpers import TOL, rel_err

pytestmark = pytest.mark.gpu


def _driven_pair(n, seed):
    """A dilute suspension in which spheres 0 and 1 start 8a apart on an axis of their own and are
    driven at each other."""
    x, _ = inputs.cube_rsa(n, 0.02, seed)
    x[:, 2] += 20.0 - x[:, 2].min()
    x[0], x[1] = (-4.0, 0.0, 0.0), (4.0, 0.1, 0.0)
    F = 0.01 * inputs.normal_forces(n, seed + 1)
    F[0], F[1] = (30.0, 0.0, 0.0), (-30.0, 0.0, 0.0)
    return x, F


@pytest.mark.parametrize("prec,n", [("fp32c", 60), ("fp32c", 300), ("fp64", 12), ("fp64", 200)])
def test_adjoint_after_steps_of_a_small_system(prec, n):
    x0, F = _driven_pair(n, 811)
    g, dt = inputs.normal_forces(n, 812), 0.02
    with sd.System(n, prec=prec) as s:
        s.set_positions(x0)
        s.set_forces(F)
        s.step(dt, 165)
        x = s.get_positions()
        assert np.linalg.norm(x[1] - x[0]) < 1.9              # overlap now; 8a apart when set
        got = s.adjoint(dt, 3, 2, g)
        np.testing.assert_array_equal(s.get_positions(), x)
    with sd.System(n, prec=prec) as s:                       # a fresh handle at these positions
        s.set_positions(x)
        s.set_forces(F)
        fresh = s.adjoint(dt, 3, 2, g)
    for a, b in zip(got, fresh):
        np.testing.assert_array_equal(a, b)
    ref = oracle.adjoint(x, F, g, 3, dt, (0.0, 0.0, 0.0))
    for a, b in zip(got, ref):
        assert rel_err(a, b) <= (1e-10 if prec == "fp64" else 1e-4)


@pytest.mark.parametrize("prec,rep", [("fp32c", 0.0), ("fp64", 0.0), ("fp64", 0.01)])
@pytest.mark.parametrize("rows", [False, True])
def test_steps_after_sharded_steps(prec, rep, rows):
    n = 2600
    x0, F = _driven_pair(n, 831)
    kw = dict(prec=prec, dense="directed" if rows else "symmetric", rep_eps=rep)
    with sd.System(n, **kw) as s:
        s.set_positions(x0)
        s.set_forces(F)
        v = s.mobility_apply(F)
        dt = 6.0 / (v[0, 0] - v[1, 0])                       # one step from 8a to 2a and less
        if rows:
            s.step_rows(dt, 0, n)
        else:
            s.step_combine(dt, s.step_part(0, 1)[None].contiguous())
        x1 = s.get_positions()
        assert 1.8 < np.linalg.norm(x1[1] - x1[0]) < 2.3
        s.step(0.1 * dt, 1)
        x2 = s.get_positions()
    with sd.System(n, **kw) as s:
        s.set_positions(x1)
        s.set_forces(F)
        s.step(0.1 * dt, 1)
        np.testing.assert_array_equal(x2, s.get_positions())
    ref = oracle.euler(x1, 1, 0.1 * dt, fext=F, rep_eps=rep, nthreads=16)
    assert np.abs(x2 - ref).max() <= 10 * TOL[prec] * np.abs(ref - x1).max()
