"""sd_set_adjoint_keep: with no bytes to keep, the adjoint's memory is what ckpt_every asks for, and
its results are the same bits."""
import numpy as np
import pytest

import paper_1205_6333_gb300 as sd
from paper_1205_6333_gb300 import inputs
from test_gpu_vjp_memory import _Allocator

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [300, 3300])   # (one launch a run of steps; step graphs)
def test_checkpoints_bound_the_memory_when_asked_to(n):
    x, _ = inputs.cube_rsa(n, 0.05, 891)
    g = inputs.normal_forces(n, 892)
    dt, T, K = 1e-3, 400, 20
    out, took = {}, {}
    for keep in (None, 0):
        al = _Allocator()
        h = sd.sd_create(al.config(n))
        try:
            if keep is not None:
                assert sd.lib().sd_set_adjoint_keep(h, -1) != 0
                assert sd.lib().sd_set_adjoint_keep(h, keep) == 0
            F = inputs.normal_forces(n, 893)
            gx, gF = np.empty_like(x), np.empty_like(x)
            sd.sd_set_positions(h, x.ctypes.data, 0)
            sd.sd_set_forces(h, F.ctypes.data, 0)
            before = al.bytes
            sd.sd_adjoint(h, dt, T, K, g.ctypes.data, gx.ctypes.data, gF.ctypes.data, 0)
            took[keep] = (al.bytes - before) / (24 * n)       # in position arrays
            if keep is None:                                  # lowered later: the buffer goes back
                live = len(al.live)
                assert sd.lib().sd_set_adjoint_keep(h, 0) == 0
                assert len(al.live) == live - 1
            out[keep] = gx, gF
        finally:
            sd.sd_destroy(h)
        assert not al.live
    assert took[None] >= T and took[0] <= T // K + 1 + K + 4
    for a, b in zip(out[None], out[0]):
        np.testing.assert_array_equal(a, b)
