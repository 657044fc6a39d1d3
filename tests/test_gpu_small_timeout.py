"""The small path's bounded waits for the other clusters' positions: with a limit of one poll they
run out, the clusters leave together, the call reports SD_ERR_TIMEOUT, and the handle then gives
the same bits as a fresh one.  Sizes with a partly filled last block (some of its cluster's CTAs
update no row) and with whole blocks, one and several CTAs per cluster."""
import numpy as np
import pytest

import paper_1205_6333_gb300 as sd
from paper_1205_6333_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,n", [("fp32c", 130), ("fp32c", 1000), ("fp32c", 1024), ("fp32c", 2011), ("fp64", 17),
                                    ("fp64", 33), ("fp64", 200), ("fp64", 1001)])
def test_small_path_wait_runs_out_and_handle_recovers(prec, n):
    x, _ = inputs.cube_rsa(n, 0.05, 841)
    F = inputs.normal_forces(n, 842)
    with sd.System(n, prec=prec) as s:
        s.set_positions(x)
        s.set_forces(F)
        s.step(0.01, 40)
        ref = s.get_positions()
    with sd.System(n, prec=prec) as s:
        s.set_forces(F)
        for _ in range(2):
            s.set_positions(x)
            s.set_watchdog(1)
            s.step(0.01, 40)
            with pytest.raises(sd.SDError) as ei:
                s.synchronize()
            assert ei.value.status_name == "SD_ERR_TIMEOUT"
            s.synchronize()                        # the error word was cleared when reported
            s.set_watchdog(1 << 22)
            s.set_positions(x)
            s.step(0.01, 40)
            np.testing.assert_array_equal(s.get_positions(), ref)
