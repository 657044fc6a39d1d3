"""The FP64 batched kernel at the edges of its 32-particle blocks and of the widths of a
partly filled last block, every launch shape, with overlapping pairs, against the FP64
oracle (steps of a few FP64 roundings: 1e-12 of the displacement, as every FP64 gate)."""
import numpy as np
import pytest

import oracle
import paper_1205_6333_gb300 as sd
from paper_1205_6333_gb300 import inputs

pytestmark = pytest.mark.gpu

SIZES = [1, 2, 3, 4, 5, 8, 9, 16, 17, 31, 32, 33, 34, 40, 48, 49, 64, 65, 96, 100, 127, 128, 129, 200, 255, 256, 0, 7]


@pytest.mark.parametrize("tensor", ["rpy", "rp", "oseen"])
def test_fp64_batch_edges_every_shape(tensor):
    sizes = np.array(SIZES, dtype=np.int32)
    x, off = inputs.ball_rsa_batch(sizes, 0.08, 71)
    for c in range(len(sizes)):          # one overlapping pair in every cluster that has two
        if sizes[c] >= 2:
            x[off[c] + 1] = x[off[c]] + np.array([0.9, 0.8, -0.4])
    F = inputs.normal_forces(x.shape[0], 72)
    ref = x.copy()
    for c in range(len(sizes)):
        if sizes[c]:
            ref[off[c]:off[c + 1]] = oracle.euler(x[off[c]:off[c + 1]], 2, 0.01, fext=F[off[c]:off[c + 1]], tensor=tensor)
    b = sd.Batch(off, prec="fp64", tensor=tensor)
    try:
        b.set_forces(F)
        for k in range(len(b.shapes())):
            b.set_shape(k)
            b.set_positions(x)
            b.step(0.01, 2)
            got = b.get_positions()
            assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref - x).max(), b.shapes()[k]
    finally:
        b.close()
