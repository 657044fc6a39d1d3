"""The one-launch path of small systems (csrc/small.cu) at the edges of its shapes, against
the FP64 oracle: one CTA / several clusters, one and two targets per thread, partly
filled blocks and splits, overlapping pairs, more near pairs than a CTA notes."""
import numpy as np
import pytest

import oracle
import paper_1205_6333_gb300 as sd
from paper_1205_6333_gb300 import inputs
from helpers import TOL, rel_err, system_with_overlaps

pytestmark = pytest.mark.gpu

# FP32C: one CTA up to 128; FP64: up to 16; last sizes before the symmetric kernels
EDGES = [("fp32c", n) for n in (1, 2, 31, 33, 65, 96, 128, 129, 255, 1021, 2047, 2048)] + \
        [("fp64", n) for n in (1, 2, 3, 5, 8, 16, 17, 33, 100, 1000, 1024)]


@pytest.mark.parametrize("prec,n", EDGES)
@pytest.mark.parametrize("tensor", ["rpy", "oseen"])
def test_small_systems_match_oracle(prec, n, tensor):
    x = system_with_overlaps(n, 0.05, seed=900 + n, overlaps=min(3, n // 2))[0] if tensor == "rpy" else \
        inputs.cube_rsa(n, 0.05, 900 + n)[0]
    F = inputs.normal_forces(n, 901 + n)
    steps, dt = 5, 0.02
    with sd.System(n, prec=prec, tensor=tensor) as s:
        s.set_positions(x)
        v = s.mobility_apply(F)
        v32 = s.mobility_apply(F.astype(np.float32))
        rows = s.mobility_apply_rows(F, n // 3, n)
        s.set_forces(F)
        s.step(dt, steps)
        x1 = s.get_positions()
        s.set_positions(x)
        for _ in range(steps):
            s.step(dt, 1)
        x2 = s.get_positions()
    ref = oracle.mobility_apply(x, F, tensor)
    assert rel_err(v, ref) <= TOL[prec]
    assert rel_err(v32, oracle.mobility_apply(x, F.astype(np.float32).astype(np.float64), tensor)) <= 1e-5
    np.testing.assert_array_equal(rows, v[n // 3:])          # a row shard: the same bits
    np.testing.assert_array_equal(x1, x2)                    # any split into launches: the same bits
    xr = oracle.euler(x, steps, dt, fext=F, tensor=tensor)
    assert np.abs(x1 - xr).max() <= 10 * TOL[prec] * np.abs(xr - x).max()


@pytest.mark.parametrize("n", [128, 700])
def test_more_near_pairs_than_a_cta_notes(n):
    """Spheres crowded into a small ball: nearly every pair is closer than r_near, far more
    than a CTA's 512 notes, and most overlap."""
    rng = np.random.default_rng(77)
    g = rng.standard_normal((n, 3))
    x = 2.0 * g / np.linalg.norm(g, axis=1)[:, None] * rng.uniform(0.2, 1.0, (n, 1))
    F = inputs.normal_forces(n, 78)
    with sd.System(n) as s:
        s.set_positions(x)
        v = s.mobility_apply(F)
        np.testing.assert_array_equal(v, s.mobility_apply(F))
    assert rel_err(v, oracle.mobility_apply(x, F, "rpy")) <= TOL["fp32c"]


@pytest.mark.parametrize("prec", ["fp32c", "fp64"])
def test_small_coincident_spheres(prec):
    x, _ = inputs.cube_rsa(60, 0.05, 91)
    x[7] = x[3]
    F = inputs.normal_forces(60, 92)
    with sd.System(60, prec=prec) as s:
        s.set_positions(x)
        assert rel_err(s.mobility_apply(F), oracle.mobility_apply(x, F, "rpy")) <= TOL[prec]
    with sd.System(60, prec=prec, tensor="rp") as s:
        s.set_positions(x)
        with pytest.raises(sd.SDError) as ei:
            s.mobility_apply(F)
        assert ei.value.status_name == "SD_ERR_COINCIDENT"


def test_small_periodic_steps_match_oracle():
    n = 500
    x, L = inputs.cube_rsa(n, 0.05, 93)
    box = (L + 2.5, 0.0, L + 2.5)
    fe = inputs.normal_forces(n, 94)
    with sd.System(n, prec="fp64", box=box) as s:
        s.set_positions(x)
        s.set_forces(fe)
        s.step(0.01, 20)
        got = s.get_positions()
    ref = oracle.euler(x, 20, 0.01, fext=fe, box=box)
    assert np.abs(got - ref).max() <= 1e-10 * np.abs(ref - x).max()
