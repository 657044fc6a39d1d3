"""The work a user of this library has it do, as cases to time and to compare.

Every case goes through the public entry points (``System``, ``Batch``,
``sd_mobility_apply_noalloc``) with CUDA tensors on torch's current stream.  The
families, and the sizes they cover:

  apply       velocities for given forces, N = 200 .. 262,144
  trajectory  Euler steps from given positions, N = 4 .. 20,000
  batch       Euler steps of many independent clusters of 4 .. 256 spheres
  adjoint     gradients through a checkpointed trajectory, N = 200 .. 4,096
  vjp         one vector-Jacobian product, N = 200 .. 16,384
  noalloc     velocities without any GPU allocation, N = 200 .. 65,536

FP32C results carry FP32 accuracy.  Where the entry point hands them out as float64
velocities or gradients they are kept as float32, as a user's program stores them;
positions are the FP64 state and stay float64.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1205_6333_gb300 as sd
from paper_1205_6333_gb300 import inputs

F64 = torch.float64


def listed():
    return [
        # The four-sphere cluster of Sec. 4: the smallest system, many steps, FP64 (the
        # paper follows its orbit for millions of steps).
        {"name": "four_spheres_fp64", "family": "trajectory", "n": 4, "prec": "fp64", "tensor": "rpy", "start": "tory",
         "steps": 512, "dt": 0.01, "gravity": True, "box": False, "rep": False, "lub": False},
        # An outer integrator that moves the particles itself (a midpoint or Brownian
        # scheme) and asks for velocities at each of its positions: a small product.
        {"name": "apply_moved_1000", "family": "apply", "n": 1000, "prec": "fp32c", "tensor": "rpy", "phi": 0.05,
         "moved": True, "box": False},
        # A small sedimenting suspension, an odd number of spheres.
        {"name": "sediment_1021", "family": "trajectory", "n": 1021, "prec": "fp32c", "tensor": "rpy", "start": "rsa",
         "phi": 0.05, "steps": 100, "dt": 0.001, "gravity": True, "box": False, "rep": False, "lub": False},
        # A lattice in a periodic box with every nearest pair in the lubrication window (the
        # paper's benchmark, Sec. 3.3, at a spacing where the friction with lagged
        # velocities grows rounding errors only slowly).
        {"name": "lubrication_4913", "family": "trajectory", "n": 4913, "prec": "fp32c", "tensor": "rpy",
         "start": "lattice", "steps": 12, "dt": 0.001, "gravity": True, "box": True, "rep": False, "lub": True},
        # A dense suspension with gravity and soft repulsion (the time-stepping workload).
        {"name": "repulsion_16384", "family": "trajectory", "n": 16384, "prec": "fp32c", "tensor": "rpy",
         "start": "rsa", "phi": 0.10, "steps": 20, "dt": 0.001, "gravity": True, "box": False, "rep": True,
         "lub": False},
        # The headline product: N = 65,536, float32 forces.
        {"name": "apply_65536", "family": "apply", "n": 65536, "prec": "fp32c", "tensor": "rpy", "phi": 0.05,
         "moved": False, "box": False},
        # The largest size of the N sweep.
        {"name": "apply_262144", "family": "apply", "n": 262144, "prec": "fp32c", "tensor": "rpy", "phi": 0.05,
         "moved": False, "box": False},
        # The reference precision, for checking FP32C results at a mid size.
        {"name": "apply_fp64_8192", "family": "apply", "n": 8192, "prec": "fp64", "tensor": "rpy", "phi": 0.05,
         "moved": False, "box": False},
        # Thousands of independent clusters (the batched workload).
        {"name": "batch_16384", "family": "batch", "clusters": 16384, "lo": 4, "hi": 256, "prec": "fp32c",
         "tensor": "rpy", "steps": 16, "dt": 0.01},
        # A batch in the reference precision.
        {"name": "batch_fp64_1000", "family": "batch", "clusters": 1000, "lo": 4, "hi": 256, "prec": "fp64",
         "tensor": "rpy", "steps": 4, "dt": 0.01},
        # Gradients with respect to the start positions and the forces through a
        # checkpointed trajectory (the differentiation workload, fewer steps).
        {"name": "adjoint_4096", "family": "adjoint", "n": 4096, "prec": "fp32c", "tensor": "rpy", "phi": 0.05,
         "steps": 40, "ckpt": 20, "dt": 0.01},
        # A caller that must not allocate (a graph under capture, a fixed memory budget).
        {"name": "noalloc_20011", "family": "noalloc", "n": 20011, "tensor": "rpy", "phi": 0.05},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    family = rng.choice(["apply", "apply", "trajectory", "trajectory", "batch", "adjoint", "vjp", "noalloc"])
    tensor = rng.choice(["rpy", "rpy", "rpy", "rp", "oseen"])
    prec = rng.choice(["fp32c", "fp32c", "fp32c", "fp64"])
    phi = round(rng.uniform(0.02, 0.12), 4)
    if family == "apply":
        n = _log_int(rng, 200, 12000 if prec == "fp64" else 100000)
        return {"family": family, "n": n, "prec": prec, "tensor": tensor, "phi": phi, "moved": rng.random() < 0.5,
                "box": rng.random() < 0.25}
    if family == "trajectory":
        n = _log_int(rng, 4, 3000 if prec == "fp64" else 20000)
        kind = rng.choice(["plain", "plain", "rep", "lub"])
        return {"family": family, "n": n, "prec": prec, "tensor": tensor,
                "start": "lattice" if kind == "lub" else "rsa", "phi": phi,
                "steps": rng.randint(4, 12 if kind == "lub" else 40), "dt": 0.001, "gravity": True, "box": rng.random() < 0.25 and n >= 200,
                "rep": kind == "rep", "lub": kind == "lub"}
    if family == "batch":
        lo = rng.randint(1, 64)
        c = _log_int(rng, 8, 1000 if prec == "fp64" else 8000)
        return {"family": family, "clusters": c, "lo": lo, "hi": rng.randint(lo, 256), "prec": prec, "tensor": tensor,
                "steps": rng.randint(1, 20) if prec == "fp32c" else rng.randint(1, 4), "dt": 0.01}
    if family == "adjoint":
        n = _log_int(rng, 200, 1500 if prec == "fp64" else 4096)
        steps = rng.randint(4, 24)
        return {"family": family, "n": n, "prec": prec, "tensor": tensor, "phi": phi, "steps": steps,
                "ckpt": rng.randint(2, steps), "dt": 0.01}
    if family == "vjp":
        n = _log_int(rng, 200, 4096 if prec == "fp64" else 16384)
        return {"family": family, "n": n, "prec": prec, "tensor": tensor, "phi": phi, "box": rng.random() < 0.25}
    return {"family": family, "n": _log_int(rng, 200, 65536), "tensor": tensor, "phi": phi}


# ---------------------------------------------------------------- inputs

def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _start(case, seed):
    """(positions n x 3, box side or None) as numpy FP64."""
    n = case["n"]
    start = case.get("start", "rsa")
    rng = np.random.default_rng(seed)
    if start == "tory":   # the orbit's start, each coordinate off by up to 0.01a
        return inputs.tory_four_spheres() + rng.uniform(-0.01, 0.01, size=(4, 3)), None
    if start == "lattice":   # simple cubic, spacing 2.9a, each coordinate off by up to 0.04a
        # (an odd number of sites a side: no separation near half a box, where the nearest
        # image of a pair is a matter of rounding)
        m = math.ceil(n ** (1.0 / 3.0) - 1e-9) | 1
        x = 2.9 * np.stack(np.meshgrid(*[np.arange(m)] * 3, indexing="ij"), -1).reshape(-1, 3)[:n]
        return x + rng.uniform(-0.04, 0.04, size=x.shape), 2.9 * m
    return inputs.cube_rsa(n, case["phi"], seed)


def _box(case, L):
    return (L, L, L) if case.get("box") else None


def _clusters(case, seed):
    """Clusters of lo .. hi spheres at volume fraction 0.05 without overlap: each is the
    neighbourhood of a random point in one large random suspension, about the origin."""
    C, lo, hi = case["clusters"], case["lo"], case["hi"]
    sizes = inputs.cluster_sizes(C, lo, hi, inputs.SEED_BASE + C)   # the same batch shape for every seed
    x, L = inputs.cube_rsa(20000, 0.05, seed + 1)
    dev = _dev()
    xs = torch.as_tensor(x, device=dev)
    edge = inputs.ball_radius(256, 0.05) + 1.0
    cen = torch.as_tensor(np.random.default_rng(seed + 2).uniform(edge, L - edge, size=(C, 3)), device=dev)
    out = []
    for c0 in range(0, C, 4096):
        c = cen[c0:c0 + 4096]
        idx = torch.cdist(c, xs).topk(hi, dim=1, largest=False, sorted=True).indices
        out.append(xs[idx] - c[:, None, :])
    full = torch.cat(out)
    keep = torch.arange(hi, device=dev)[None, :] < torch.as_tensor(sizes.astype(np.int64), device=dev)[:, None]
    off = np.zeros(C + 1, dtype=np.int32)
    off[1:] = np.cumsum(sizes)
    return full[keep].contiguous(), off, sizes


def _forces(n, seed, dtype=F64):
    return torch.as_tensor(inputs.normal_forces(n, seed + 7), device=_dev(), dtype=dtype).contiguous()


def _gravity(case):
    return (0.0, 0.0, -1.0) if case.get("gravity") else (0.0, 0.0, 0.0)


def prepare(case, seed):
    f = case["family"]
    dev = _dev()
    if f == "batch":
        x, off, _ = _clusters(case, seed)
        b = sd.Batch(off, tensor=case["tensor"], prec=case["prec"], stream="torch")
        b.set_forces(_forces(x.shape[0], seed))
        return {"case": case, "b": b, "x": x, "out": torch.empty_like(x)}
    xn, L = _start(case, seed)
    x = torch.as_tensor(xn, device=dev, dtype=F64).contiguous()
    n = x.shape[0]
    if f == "noalloc":
        return {"case": case, "x": x, "F": _forces(n, seed), "V": torch.empty_like(x)}
    s = sd.System(n, tensor=case["tensor"], prec=case["prec"], stream="torch", box=_box(case, L),
                  gravity=_gravity(case) if f == "trajectory" else ((0.0, 0.0, -1.0) if f == "adjoint" else (0.0,) * 3),
                  rep_eps=1.0 if case.get("rep") else 0.0, lubrication=bool(case.get("lub")))
    st = {"case": case, "s": s, "x": x}
    work = torch.float32 if case["prec"] == "fp32c" else F64
    if f == "apply":
        st["F"] = _forces(n, seed, work)
        s.set_positions(x)
    elif f == "vjp":
        st["F"] = _forces(n, seed, work)
        st["W"] = _forces(n, seed + 1, work)
        s.set_positions(x)
    elif f == "adjoint":
        st["F"] = 0.1 * _forces(n, seed)
        st["g"] = _forces(n, seed + 1)
        s.set_positions(x)
        s.set_forces(st["F"])
    else:
        st["out"] = torch.empty_like(x)
    return st


def run(state):
    case = state["case"]
    f = case["family"]
    if f == "apply":
        s = state["s"]
        if case["moved"]:
            s.set_positions(state["x"])
        return s.mobility_apply(state["F"])
    if f == "trajectory":
        s = state["s"]
        s.set_positions(state["x"])
        s.step(case["dt"], case["steps"])
        return s.get_positions(state["out"])
    if f == "batch":
        b = state["b"]
        b.set_positions(state["x"])
        b.step(case["dt"], case["steps"])
        return b.get_positions(state["out"])
    if f == "adjoint":
        gx, gF = state["s"].adjoint(case["dt"], case["steps"], case["ckpt"], state["g"])
        return (gx.float(), gF.float()) if case["prec"] == "fp32c" else (gx, gF)
    if f == "vjp":
        return state["s"].vjp(state["F"], state["W"])
    x, V = state["x"], state["V"]
    sd.sd_mobility_apply_noalloc(x.data_ptr(), state["F"].data_ptr(), V.data_ptr(), x.shape[0], 1.0, 1.0,
                                 case["tensor"], torch.cuda.current_stream().cuda_stream)
    return V.float()


def _pairs(case):
    """Unordered pairs of one evaluation, and the spheres."""
    if case["family"] == "batch":
        k = np.arange(case["lo"], case["hi"] + 1, dtype=np.float64)
        return case["clusters"] * float((k * (k - 1) / 2).mean()), case["clusters"] * float(k.mean())
    n = case["n"]
    return n * (n - 1) / 2.0, float(n)


def work(case):
    """The floating-point operations of one pass with every unordered pair once: 53 a
    pair for the product (separation 3, r^2 5, 1/r 1, the tensor's two scalars 8, and 18
    for each direction), 118 with the vector-Jacobian product's two sums; inputs read once
    and outputs written once."""
    p, n = _pairs(case)
    f = case["family"]
    es = 4 if case.get("prec") == "fp32c" else 8
    if f == "apply":
        return {"bytes": n * 3 * (8 + 2 * es), "flops": 53 * p}
    if f == "noalloc":
        return {"bytes": n * 3 * 24, "flops": 53 * p}
    if f == "vjp":
        return {"bytes": n * 3 * (8 + 4 * es), "flops": 118 * p}
    if f == "adjoint":
        return {"bytes": n * 3 * 8 * 5, "flops": case["steps"] * (53 + 118) * p}
    return {"bytes": n * 3 * 8 * 3, "flops": case["steps"] * 53 * p}


# ---------------------------------------------------------------- exact values (plain torch, FP64)

MU0 = 1.0 / (6.0 * math.pi)


def _profile(r2, tensor):
    """A, B of T / mu0 = A I + B r r^T; the caller masks the self pairs (r = 0)."""
    r2 = torch.where(r2 > 0, r2, torch.full_like(r2, 1.0))
    ri = r2.rsqrt()
    ri3 = ri / r2
    if tensor == "oseen":
        return 0.75 * ri, 0.75 * ri3
    A = 0.75 * ri + 0.5 * ri3
    B = 0.75 * ri3 - 1.5 * ri3 / r2
    if tensor == "rpy":
        near = r2 < 4.0
        A = torch.where(near, 1.0 - (9.0 / 32.0) * r2 * ri, A)
        B = torch.where(near, (3.0 / 32.0) * ri, B)
    return A, B


def _image(d, L):
    return d if L is None else d - L * torch.round(d / L)


def _rows(n):
    return max(1, min(n, 20_000_000 // max(n, 1)))


def _velocities(x, F, tensor, L=None):
    n = x.shape[0]
    v = torch.empty_like(F)
    for i0 in range(0, n, _rows(n)):
        i1 = min(n, i0 + _rows(n))
        d = [_image(x[i0:i1, k, None] - x[None, :, k], L) for k in range(3)]
        A, B = _profile(d[0] * d[0] + d[1] * d[1] + d[2] * d[2], tensor)
        k = torch.arange(i0, i1, device=x.device)
        A[k - i0, k] = 1.0
        B[k - i0, k] = 0.0
        s = B * (d[0] * F[:, 0] + d[1] * F[:, 1] + d[2] * F[:, 2])
        for c in range(3):
            v[i0:i1, c] = (A * F[:, c] + s * d[c]).sum(1)
    return MU0 * v


def _pair_forces(x, vlag, case, L):
    """Soft repulsion (eps = 1, cut at 2.5a) and the lubrication friction with the
    previous velocities, for every sphere."""
    n = x.shape[0]
    f = torch.zeros_like(x)
    for i0 in range(0, n, _rows(n)):
        i1 = min(n, i0 + _rows(n))
        d = [_image(x[i0:i1, k, None] - x[None, :, k], L) for k in range(3)]
        i, j = torch.nonzero(d[0] * d[0] + d[1] * d[1] + d[2] * d[2] < 9.0, as_tuple=True)
        other = i + i0 != j
        i, j = i[other], j[other]
        e = torch.stack([d[k][i, j] for k in range(3)], 1)
        i = i + i0
        r = e.square().sum(1).sqrt()
        t = torch.zeros_like(e)
        if case["rep"]:
            t += torch.where(r < 2.5, 12.0 * 2.0 ** 12 / r ** 14, torch.zeros_like(r))[:, None] * e
        if case["lub"]:
            e = e / r[:, None]
            s = r - 2.0
            on = (s > 0) & (s < 1)
            ls = torch.log(torch.where(on, s, torch.ones_like(s)))
            zn = 0.25 / torch.where(on, s, torch.ones_like(s)) - 0.225 * ls
            zt = -ls / 6.0
            w = vlag[i] - vlag[j]
            en = (e * w).sum(1)
            t -= torch.where(on[:, None], ((zn - zt) * en)[:, None] * e + zt[:, None] * w, torch.zeros_like(w)) / MU0
        f.index_add_(0, i, t)
    return f


def _exact_batch(case, seed):
    x, off, sizes = _clusters(case, seed)
    F = _forces(x.shape[0], seed)
    dev, m = x.device, int(case["hi"])
    n = torch.as_tensor(sizes.astype(np.int64), device=dev)
    here = torch.arange(m, device=dev)[None, :] < n[:, None]
    X = torch.zeros((len(sizes), m, 3), dtype=F64, device=dev)
    G = torch.zeros_like(X)
    X[here] = x
    G[here] = F
    eye = torch.eye(m, dtype=torch.bool, device=dev)[None]
    per = max(1, 20_000_000 // (m * m))
    for c0 in range(0, len(sizes), per):
        xc, gc = X[c0:c0 + per], G[c0:c0 + per]
        for _ in range(case["steps"]):
            d = [xc[:, :, None, k] - xc[:, None, :, k] for k in range(3)]
            A, B = _profile(d[0] * d[0] + d[1] * d[1] + d[2] * d[2], case["tensor"])
            A = A.masked_fill(eye, 1.0)
            B = B.masked_fill(eye, 0.0)
            s = B * (d[0] * gc[:, None, :, 0] + d[1] * gc[:, None, :, 1] + d[2] * gc[:, None, :, 2])
            v = torch.stack([(A * gc[:, None, :, k] + s * d[k]).sum(2) for k in range(3)], 2)
            xc = xc + case["dt"] * MU0 * v
        X[c0:c0 + per] = xc
    return X[here]


def _exact_vjp(x, F, W, tensor, L=None):
    """Gradients of sum_i W_i . v_i with respect to x and F."""
    n = x.shape[0]
    gx, gF = torch.zeros_like(x), torch.zeros_like(F)
    step = max(1, _rows(n) // 4)
    for i0 in range(0, n, step):
        i1 = min(n, i0 + step)
        xs, Fs = x.detach().requires_grad_(), F.detach().requires_grad_()
        d = [_image(xs[i0:i1, k, None] - xs[None, :, k], L) for k in range(3)]
        A, B = _profile(d[0] * d[0] + d[1] * d[1] + d[2] * d[2], tensor)
        me = torch.zeros((i1 - i0, n), dtype=torch.bool, device=x.device)
        k = torch.arange(i0, i1, device=x.device)
        me[k - i0, k] = True
        A = A.masked_fill(me, 1.0)
        B = B.masked_fill(me, 0.0)
        Wr = W[i0:i1]
        wd = d[0] * Wr[:, 0, None] + d[1] * Wr[:, 1, None] + d[2] * Wr[:, 2, None]
        fd = d[0] * Fs[:, 0] + d[1] * Fs[:, 1] + d[2] * Fs[:, 2]
        S = MU0 * ((A * (Wr @ Fs.T)).sum() + (B * wd * fd).sum())
        a, b = torch.autograd.grad(S, (xs, Fs))
        gx += a
        gF += b
    return gx, gF


def exact(case, seed):
    f = case["family"]
    if f == "batch":
        return _exact_batch(case, seed)
    if case["n"] > 131072:
        return None
    xn, side = _start(case, seed)
    x = torch.as_tensor(xn, device=_dev(), dtype=F64)
    n, t = x.shape[0], case["tensor"]
    L = side if case.get("box") else None
    if f in ("apply", "noalloc"):
        F = _forces(n, seed, torch.float32 if case.get("prec") == "fp32c" else F64)
        return _velocities(x, F.double(), t, L)
    if f == "vjp":
        work = torch.float32 if case["prec"] == "fp32c" else F64
        return _exact_vjp(x, _forces(n, seed, work).double(), _forces(n, seed + 1, work).double(), t, L)
    dt = case["dt"]
    g = torch.tensor([0.0, 0.0, -1.0], dtype=F64, device=x.device)
    if f == "trajectory":
        v = torch.zeros_like(x)
        for _ in range(case["steps"]):
            F = g.expand(n, 3).clone()
            if case["rep"] or case["lub"]:
                F += _pair_forces(x, v, case, L)
            v = _velocities(x, F, t, L)
            x = x + dt * v
        return x
    F = 0.1 * _forces(n, seed) + g
    xs = [x]
    for _ in range(case["steps"]):
        xs.append(xs[-1] + dt * _velocities(xs[-1], F, t))
    lam, gF = _forces(n, seed + 1), torch.zeros_like(x)
    for k in range(case["steps"] - 1, -1, -1):
        a, b = _exact_vjp(xs[k], F, lam, t)
        lam, gF = lam + dt * a, gF + dt * b
    return lam, gF
