"""Systems around the size from which the symmetric kernel takes over from the one-launch path
(3,072 in FP32C and 1,408 in FP64 on 152 SMs), against the oracle."""
import numpy as np
import pytest

import oracle
import paper_1205_6333_gb300 as sd
from paper_1205_6333_gb300 import inputs
from helpers import TOL, periodic_rel_err, rel_err, system_with_overlaps

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,n", [("fp32c", 2049), ("fp32c", 2500), ("fp32c", 3071), ("fp32c", 3072), ("fp32c", 3073),
                                    ("fp64", 1025), ("fp64", 1250), ("fp64", 1407), ("fp64", 1408), ("fp64", 1409)])
@pytest.mark.parametrize("box", [False, True])
def test_either_side_of_the_small_path_limit(prec, n, box):
    x, L = system_with_overlaps(n, 0.05, seed=931 + n)
    F = inputs.normal_forces(n, 932)
    kw = dict(box=(0.0, L + 2.5, 0.0)) if box else {}
    with sd.System(n, prec=prec, **kw) as s:
        s.set_positions(x)
        v = s.mobility_apply(F)
        s.set_forces(F)
        s.step(0.01, 3)
        x1 = s.get_positions()
        s.set_positions(x)
        for _ in range(3):
            s.step(0.01, 1)
        np.testing.assert_array_equal(s.get_positions(), x1)
    ref = oracle.mobility_apply(x, F, "rpy", nthreads=16, **kw)
    if box and prec == "fp32c":   # (which image of a pair near half a period is the nearer is a matter of FP32 rounding)
        assert periodic_rel_err(v, ref, x, F, kw["box"]) <= TOL[prec]
        return
    assert rel_err(v, ref) <= TOL[prec]
    ref = oracle.euler(x, 3, 0.01, fext=F, nthreads=16, **kw)
    assert np.abs(x1 - ref).max() <= 10 * TOL[prec] * np.abs(ref - x).max()
