"""Products whose output overlaps their input (V = F, or rows of V inside F): every path stages or
copies the forces it still reads.  The CTAs of a launch are spread in time, by near pairs that some
have far more of than others and by another stream's work, so that a direct read would see results."""
import numpy as np
import pytest

import paper_1205_6333_gb300 as sd
from paper_1205_6333_gb300 import inputs

pytestmark = pytest.mark.gpu


def _crowded(n, seed):
    """A dilute suspension; with 300 spheres or more, four of the first block and 150 of later ones in one small ball."""
    x, _ = inputs.cube_rsa(n, 0.02, seed)
    if n >= 300:
        rng = np.random.default_rng(seed + 1)
        idx = np.concatenate([np.arange(4), np.arange(100, 250)])
        g = rng.standard_normal((idx.size, 3))
        x[idx] = x.min() - 30.0 + 2.0 * g / np.linalg.norm(g, axis=1)[:, None] * rng.uniform(0.2, 1.0, (idx.size, 1))
    return x


@pytest.mark.parametrize("prec,n", [("fp32c", 5), ("fp32c", 300), ("fp32c", 2000), ("fp32c", 4000), ("fp64", 16),
                                    ("fp64", 300), ("fp64", 1024), ("fp64", 2000)])
@pytest.mark.parametrize("dtype", [0, 1])
def test_product_in_place(prec, n, dtype):
    import torch
    x = _crowded(n, 851)
    F = torch.tensor(inputs.normal_forces(n, 852), device="cuda",
                     dtype=torch.float32 if dtype == 0 else torch.float64)
    code = sd.SD_DTYPE_F32 if dtype == 0 else sd.SD_DTYPE_F64
    other, m = torch.cuda.Stream(), torch.randn(4096, 4096, device="cuda")
    with sd.System(n, prec=prec, stream="torch") as s:
        s.set_positions(x)
        ref = s.mobility_apply(F)
        rows = s.dense_kernel() == "directed" and n > 5
        torch.cuda.synchronize()
        for _ in range(20):
            with torch.cuda.stream(other):
                m @ m
            b = F.clone()
            sd.sd_mobility_apply(s.h, b.data_ptr(), b.data_ptr(), code, 1)
            assert torch.equal(b, ref)
            if rows:
                r0 = n // 3
                c = torch.cat([F, torch.zeros_like(F)])
                out = c[3:3 + n - r0]                        # rows r0 .. n-1, written over rows of F
                sd.sd_mobility_apply_rows(s.h, c.data_ptr(), out.data_ptr(), code, 1, r0, n)
                assert torch.equal(out, ref[r0:])
