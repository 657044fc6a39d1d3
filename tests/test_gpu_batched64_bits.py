"""FP64 batches: the launch shape, which the autotuner picks by timing, does not change a bit."""
import numpy as np
import pytest

import paper_1205_6333_gb300 as sd
from paper_1205_6333_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tensor", ["rpy", "oseen"])
def test_every_launch_shape_gives_the_same_bits(tensor):
    sizes = np.array([256, 255, 129, 128, 100, 97, 96, 65, 64, 33, 32, 5, 1, 0, 200, 161], dtype=np.int32)
    x, off = inputs.ball_rsa_batch(sizes, 0.08, 871)
    F = inputs.normal_forces(x.shape[0], 872)
    got = {}
    b = sd.Batch(off, prec="fp64", tensor=tensor)
    try:
        b.set_forces(F)
        for k, shape in enumerate(b.shapes()):
            b.set_shape(k)
            b.set_positions(x)
            b.step(0.01, 3)
            got.setdefault(shape["threads"], []).append(b.get_positions())
    finally:
        b.close()
    assert len(got) > 1
    ref = next(iter(got.values()))[0]
    for many in got.values():
        for y in many:
            np.testing.assert_array_equal(y, ref)
