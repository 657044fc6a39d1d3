"""Vector-Jacobian products at the edges of the kernels' blocks, and above the size from which
the directed kernels run, against the oracle and a plain torch FP64 sum.  Bounds as in
test_gpu_vjp.py."""
import numpy as np
import pytest

import oracle
import paper_1205_6333_gb300 as sd
from paper_1205_6333_gb300 import inputs
from helpers import rel_err, system_with_overlaps

pytestmark = pytest.mark.gpu


def _check(x, n, tensor, prec, box=None):
    F, W = inputs.normal_forces(n, 72 + n), inputs.normal_forces(n, 73 + n)
    with sd.System(n, tensor=tensor, prec=prec, **({"box": box} if box else {})) as s:
        s.set_positions(x)
        gx, gF = s.vjp(F, W)
    rx, rF = oracle.vjp(x, F, W, tensor, box=box, nthreads=16)
    tol = 1e-11 if prec == "fp64" else 1e-5
    assert rel_err(gF, rF) <= tol
    if np.abs(rx).max() > 0:
        assert rel_err(gx, rx) <= 10 * tol


@pytest.mark.parametrize("tensor", ["rpy", "oseen"])
@pytest.mark.parametrize("prec,n", [("fp32c", 1), ("fp32c", 63), ("fp32c", 65), ("fp32c", 3712), ("fp32c", 3841),
                                    ("fp64", 2), ("fp64", 33), ("fp64", 97), ("fp64", 3905)])
def test_vjp_at_block_edges(prec, n, tensor):
    x = system_with_overlaps(n, 0.05, seed=71 + n, overlaps=4)[0] if n > 20 else inputs.cube_rsa(n, 0.05, 71 + n)[0]
    _check(x, n, tensor, prec)


@pytest.mark.parametrize("prec,m", [("fp32c", 15), ("fp32c", 17), ("fp64", 13)])
def test_vjp_periodic(prec, m):
    # an odd lattice: no separation is near half a box, where FP32 could take the other image
    x = 2.4 * np.stack(np.meshgrid(*[np.arange(m)] * 3, indexing="ij"), -1).reshape(-1, 3)
    x = x + np.random.default_rng(74).uniform(-0.04, 0.04, size=x.shape)
    _check(x, m ** 3, "rpy", prec, (2.4 * m,) * 3)


@pytest.mark.parametrize("prec,n", [("fp32c", 15617), ("fp32c", 65537), ("fp64", 65537)])
def test_vjp_rows_of_large_systems(prec, n):
    import torch
    x, _ = inputs.cube_rsa(n, 0.05, 81)
    F, W = inputs.normal_forces(n, 82), inputs.normal_forces(n, 83)
    with sd.System(n, prec=prec) as s:
        s.set_positions(x)
        gx, gF = s.vjp(F, W)
    rows = np.sort(np.random.default_rng(84).choice(n, 64, replace=False))
    xs = torch.tensor(x[rows], requires_grad=True)
    Fs, Ws = torch.tensor(F[rows]), torch.tensor(W[rows])
    X, FA, WA = torch.tensor(x), torch.tensor(F), torch.tensor(W)
    d = xs[:, None, :] - X[None]
    me = torch.zeros(len(rows), n, dtype=torch.bool)
    me[torch.arange(len(rows)), torch.tensor(rows)] = True
    r2 = (d * d).sum(2).masked_fill(me, 1.0)
    ri = r2.rsqrt()
    A = (0.75 * ri + 0.5 * ri ** 3).masked_fill(me, 0.0)
    B = (0.75 * ri ** 3 - 1.5 * ri ** 5).masked_fill(me, 0.0)

    def pair(u, v):   # sum over pairs of u_i . T v_j
        return (A * (u @ v.T) + B * (d * u[:, None, :]).sum(2) * (d * v[None]).sum(2)).sum()

    mu0 = 1.0 / (6.0 * np.pi)
    (g,) = torch.autograd.grad(mu0 * (pair(Ws, FA) + pair(Fs, WA)), xs)
    mW = mu0 * (Ws + A @ WA + ((B * (d * WA[None]).sum(2))[:, :, None] * d).sum(1))
    tol = 1e-11 if prec == "fp64" else 1e-5
    assert rel_err(gF[rows], mW.detach().numpy()) <= tol
    assert rel_err(gx[rows], g.numpy()) <= 10 * tol
