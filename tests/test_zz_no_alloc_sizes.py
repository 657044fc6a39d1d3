"""sd_mobility_apply_noalloc at the edges of its blocks, tiles and variants, against the oracle.

The bound is the FP32C one of the other GPU tests (FP32 pair terms, compensated sums).
"""
import pytest

import oracle
from paper_1205_6333_gb300 import inputs
from helpers import TOL, rel_err, system_with_overlaps
from test_zz_no_alloc import _noalloc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tensor", ["rpy", "rp", "oseen"])
@pytest.mark.parametrize("n", [1, 2, 63, 65, 129, 257, 1024, 4095, 4096, 4353])
def test_noalloc_block_and_variant_edges(n, tensor):
    x = (system_with_overlaps(n, 0.05, seed=331 + n, overlaps=2)[0] if n > 10
         else inputs.cube_rsa(n, 0.05, seed=331 + n)[0])
    F = inputs.normal_forces(n, 332 + n)
    assert rel_err(_noalloc(x, F, tensor), oracle.mobility_apply(x, F, tensor)) <= TOL["fp32c"]
