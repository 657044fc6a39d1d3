"""The VJP's partial sums: a system holds them from its creation while they are small, larger ones
from its first gradient on, which may run out of memory, or be recorded into a caller's graph."""
import numpy as np
import pytest

import paper_1205_6333_gb300 as sd
from paper_1205_6333_gb300 import inputs
from helpers import TOL, rel_err
from test_gpu_failures import _CountingAllocator

pytestmark = pytest.mark.gpu


class _Allocator(_CountingAllocator):
    """... that counts the bytes."""
    bytes = 0

    def _alloc(self, nbytes, ctx):
        p = super()._alloc(nbytes, ctx)
        self.bytes += int(nbytes) if p else 0
        return p


@pytest.mark.parametrize("n,prec,lazy", [(3000, "fp32c", False), (4096, "fp64", False), (40000, "fp32c", True),
                                         (20000, "fp64", True)])
def test_gradient_buffers_come_with_the_first_gradient(n, prec, lazy):
    x, _ = inputs.cube_rsa(n, 0.05, 881)
    F, W = inputs.normal_forces(n, 882), inputs.normal_forces(n, 883)
    al = _Allocator()
    cfg = al.config(n)
    cfg.prec = sd.PRECISIONS[prec]
    h = sd.sd_create(cfg)
    try:
        ptr = lambda a: a.ctypes.data
        V, gX, gF = np.empty_like(x), np.empty_like(x), np.empty_like(x)
        sd.sd_set_positions(h, ptr(x), 0)
        sd.sd_mobility_apply(h, ptr(W), ptr(V), sd.SD_DTYPE_F64, 0)
        sd.sd_mobility_apply(h, ptr(W), ptr(V), sd.SD_DTYPE_F64, 0)
        sd.sd_step(h, 0.0, 1)
        before, calls = al.bytes, al.calls
        if lazy:
            al.fail = True
            with pytest.raises(sd.SDError) as ei:
                sd.sd_mobility_vjp(h, ptr(F), ptr(W), ptr(gX), ptr(gF), sd.SD_DTYPE_F64, 0)
            assert ei.value.status_name == "SD_ERR_OOM"
            al.fail = False
        sd.sd_mobility_vjp(h, ptr(F), ptr(W), ptr(gX), ptr(gF), sd.SD_DTYPE_F64, 0)
        assert (al.bytes - before >= 128 << 20) == lazy       # (the calls' staging buffer is a few MB)
        now = al.bytes
        sd.sd_mobility_vjp(h, ptr(F), ptr(W), ptr(gX), ptr(gF), sd.SD_DTYPE_F64, 0)
        assert al.bytes == now
    finally:
        sd.sd_destroy(h)
    assert not al.live
    assert rel_err(gF, V) <= 2 * TOL[prec]                    # mu is symmetric
    assert np.abs(gX.sum(0)).max() <= 10 * TOL[prec] * np.abs(gX).max() * np.sqrt(n)   # a shift of all changes nothing


@pytest.mark.parametrize("n,prec", [(3000, "fp32c"), (40000, "fp32c"), (20000, "fp64")])
def test_first_gradient_inside_a_capture(n, prec):
    import torch
    x, _ = inputs.cube_rsa(n, 0.05, 885)
    F = torch.tensor(inputs.normal_forces(n, 886), device="cuda")
    W = torch.tensor(inputs.normal_forces(n, 887), device="cuda")
    gX, gF = torch.empty_like(F), torch.empty_like(F)
    st = torch.cuda.Stream()
    with sd.System(n, prec=prec) as s:
        s.set_positions(x)
        ref = s.vjp(F, W)
        torch.cuda.synchronize()
    with sd.System(n, prec=prec, stream=st.cuda_stream) as s:
        s.set_positions(x)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            sd.sd_mobility_vjp(s.h, F.data_ptr(), W.data_ptr(), gX.data_ptr(), gF.data_ptr(), sd.SD_DTYPE_F64, 1)
        for _ in range(2):
            gX.zero_(), gF.zero_()
            g.replay()
            torch.cuda.synchronize()
            assert rel_err(gF.cpu().numpy(), ref[1].cpu().numpy()) <= TOL[prec]
            assert rel_err(gX.cpu().numpy(), ref[0].cpu().numpy()) <= 10 * TOL[prec]
        del g
