"""Several live systems: a kernel's shared-memory limit belongs to the function, which all
handles share, so creating one system must not take away what another's launches ask for.
Every group holds systems that run the same kernels with different shapes (one-launch small
systems; all-pairs launches spread over the SMs; symmetric kernel here, directed there)."""
import numpy as np
import pytest

import paper_1205_6333_gb300 as sd
from paper_1205_6333_gb300 import inputs

pytestmark = pytest.mark.gpu

GROUPS = [
    [dict(n=2000), dict(n=1500), dict(n=1000), dict(n=130)],
    [dict(n=1024, prec="fp64"), dict(n=300, prec="fp64"), dict(n=10, prec="fp64")],
    [dict(n=5000, prec="fp64"), dict(n=1500, prec="fp64"), dict(n=500, prec="fp64")],
    [dict(n=3500), dict(n=1000), dict(n=8192)],
    [dict(n=1000, prec="fp64", rep_eps=0.01), dict(n=3000, prec="fp64"), dict(n=1500, rep_eps=0.01), dict(n=8192)],
]


def _run(s, n, rep):
    x, _ = inputs.cube_rsa(n, 0.05, 700 + n)
    F = inputs.normal_forces(n, 701 + n)
    s.set_positions(x)
    s.set_forces(F)
    out = [s.mobility_apply(F), *s.vjp(F, F[::-1].copy())]
    if not rep:
        out += s.adjoint(0.01, 3, 2, F)
    s.step(0.01, 3)
    return out + [s.get_positions()]


@pytest.mark.parametrize("group", range(len(GROUPS)))
@pytest.mark.parametrize("order", [1, -1])
def test_systems_of_different_sizes_side_by_side(group, order):
    kws = GROUPS[group][::order]
    alone = []
    for kw in kws:
        with sd.System(**kw) as s:
            alone.append(_run(s, kw["n"], "rep_eps" in kw))
    live = [sd.System(**kw) for kw in kws]
    try:
        for _ in range(2):
            for kw, s, ref in zip(kws, live, alone):
                for a, b in zip(_run(s, kw["n"], "rep_eps" in kw), ref):
                    np.testing.assert_array_equal(a, b)
    finally:
        for s in live:
            s.close()
