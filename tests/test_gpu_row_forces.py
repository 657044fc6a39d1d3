"""A row shard sums over all n forces, so a non-finite one is reported whichever rows are asked for."""
import numpy as np
import pytest

import paper_1205_6333_gb300 as sd
from paper_1205_6333_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,n,dense", [("fp32c", 20, "auto"), ("fp32c", 1500, "auto"), ("fp64", 10, "auto"),
                                          ("fp64", 700, "auto"), ("fp32c", 700, "directed")])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("dtype", [np.float64, np.float32])
def test_nonfinite_force_outside_the_rows_is_reported(prec, n, dense, bad, dtype):
    x, _ = inputs.cube_rsa(n, 0.05, 861)
    good = inputs.normal_forces(n, 862).astype(dtype)
    with sd.System(n, prec=prec, dense=dense) as s:
        s.set_positions(x)
        ref = s.mobility_apply(good)
        for at, r0, r1 in [(0, n // 2, n), (n - 1, 0, n // 2), (n // 2, 0, 1), (n - 1, 0, n)]:
            F = good.copy()
            F[at, 1] = bad
            with pytest.raises(sd.SDError) as ei:
                s.mobility_apply_rows(F, r0, r1)
            assert ei.value.status_name == "SD_ERR_NONFINITE"
            np.testing.assert_array_equal(s.mobility_apply_rows(good, r0, r1), ref[r0:r1])
