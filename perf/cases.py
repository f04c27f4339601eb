"""The workloads the library's speed is measured on, through its public Python entry points.

Four kinds of call carry the method (Steps 1-4 of the midpoint scheme) and its warm start:

  solve     a whole run from a raw block: ``Solver`` on device data, K time steps, U and E
  batch     the same for several uneven problems advanced together by ``Batch``
  cg        Step 1 alone: ``cg_solve`` from a zero start
  midpoint  Steps 2-4 of an FP32 block for a given W: ``gram``, ``core``, ``update``
  gram64    the FP64 inner matrices C, S, D: ``gram_fp64tc``
  update64  the FP64 rank-2p update: ``update_fp64tc``
  forward   the warm-start network V -> Y: ``Net.forward``
  gradient  its training loss and whole gradient: ``Net.loss_grad``

Inputs are drawn on the GPU from the seed: harmonic traps with Gaussian wells, raw Gaussian or
orthonormal blocks, He-uniform network weights.
"""
import math

import numpy as np
import torch

from paper_2511_06788_gb300 import binding as gb

DEV = "cuda"
LOSS_WEIGHT = 0.1  # gamma of the network's loss (the binding's default)


def listed():
    return [
        # the smallest solve: 2-D Laplace on the unit square, where launches and host
        # synchronisations are all there is
        {"name": "solve_2d_32_p8_fp64", "kind": "solve", "dim": 2, "nx": 32, "ny": 32, "nz": 1, "p": 8,
         "box": 0.5, "wells": 0, "prec": "fp64", "cg_rtol": 1e-10, "steps": 20},
        # the ordinary FP32 run: harmonic trap with wells at 64^3, 128 orbitals, Step 1 to a
        # tolerance in the middle of the default rule's range
        {"name": "solve_64c_p128_fp32", "kind": "solve", "dim": 3, "nx": 64, "ny": 64, "nz": 64, "p": 128,
         "box": 8.0, "wells": 8, "prec": "fp32", "cg_rtol": 1e-3, "steps": 20},
        # the ordinary FP64 run (tensor-core products, refinement around an FP32 CG) at an
        # oscillator-shell cut, p not a multiple of 32
        {"name": "solve_64c_p84_fp64", "kind": "solve", "dim": 3, "nx": 64, "ny": 64, "nz": 64, "p": 84,
         "box": 8.0, "wells": 8, "prec": "fp64", "cg_rtol": 1e-10, "steps": 10},
        # many small uneven problems, replayed as graphs
        {"name": "batch_16_fp32", "kind": "batch", "count": 16, "nmin": 24, "nmax": 48, "pmin": 16, "pmax": 96,
         "cg_rtol": 1e-3, "steps": 60},
        # Step 1 alone, FP32 3-D, odd axes and an odd p
        {"name": "cg_97x80x71_p100_fp32", "kind": "cg", "dim": 3, "nx": 97, "ny": 80, "nz": 71, "p": 100,
         "box": 8.0, "wells": 12, "prec": "fp32", "precond": "jacobi", "rtol": 1e-6},
        # Step 1 alone, FP64 2-D: the 199 x 199 oscillator of the paper's first test, p = 15
        {"name": "cg_199x199_p15_fp64", "kind": "cg", "dim": 2, "nx": 199, "ny": 199, "nz": 1, "p": 15,
         "box": 5.5, "wells": 0, "prec": "fp64", "precond": "none", "rtol": 1e-10},
        # Steps 2-4 of an FP32 step at 64^3 x 128
        {"name": "midpoint_262144_p128", "kind": "midpoint", "n": 262144, "p": 128},
        # the same for a ragged p (rows not a multiple of 32 columns) and an odd point count
        {"name": "midpoint_357911_p84", "kind": "midpoint", "n": 357911, "p": 84},
        # the FP64 inner matrices of a wide block, the width of the largest configuration
        {"name": "gram64_262144_p1024", "kind": "gram64", "n": 262144, "p": 1024},
        # the FP64 update on the largest grid, ragged p
        {"name": "update64_2097152_p200", "kind": "update64", "n": 2097152, "p": 200},
        # the learned warm start at 48^3 and p = 64: inference
        {"name": "net_forward_48c_p64", "kind": "forward", "N": 48, "p": 64, "c0": 24, "c1": 48, "c2": 96},
        # and one training gradient
        {"name": "net_gradient_48c_p64", "kind": "gradient", "N": 48, "p": 64, "c0": 24, "c1": 48, "c2": 96},
    ]


def draw(rng):
    def log(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    kind = rng.choice(["solve", "solve", "batch", "cg", "cg", "midpoint", "midpoint", "gram64", "gram64",
                       "update64", "update64", "forward", "gradient"])
    if kind in ("solve", "cg"):
        dim = rng.choice([2, 3, 3])
        top = 256 if dim == 2 else 72
        nx, ny, nz = log(24, top), log(24, top), (log(24, top) if dim == 3 else 1)
        p = log(4, 24) if dim == 2 else log(8, 128)
        prec = rng.choice(["fp32", "fp64"])
        c = {"kind": kind, "dim": dim, "nx": nx, "ny": ny, "nz": nz, "p": p,
             "box": 5.5 if dim == 2 else 8.0, "wells": rng.randint(0, 12), "prec": prec}
        if kind == "solve":
            c.update(cg_rtol=1e-3 if prec == "fp32" else 1e-10, steps=rng.randint(4, 12))
        else:
            c.update(precond=rng.choice(["jacobi", "none"]), rtol=1e-6 if prec == "fp32" else 1e-10)
        return c
    if kind == "batch":
        return {"kind": kind, "count": rng.randint(3, 16), "nmin": 20, "nmax": rng.randint(28, 48), "pmin": 9,
                "pmax": rng.randint(24, 96), "cg_rtol": 1e-3, "steps": rng.randint(10, 50)}
    if kind == "midpoint":
        return {"kind": kind, "n": log(4000, 500000), "p": log(8, 128)}
    if kind in ("gram64", "update64"):
        p = log(16, 1024)
        return {"kind": kind, "n": log(8000, min(2097152, 2.4e11 / p**2)), "p": p}
    N = 4 * rng.randint(4, 12)
    return {"kind": kind, "N": N, "p": 8 * rng.randint(1, 8), "c0": 24, "c1": 48, "c2": 96}


# ---- inputs -----------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _shape(case):
    return (case["nx"], case["ny"], case["nz"])[: case["dim"]]


def _potential(shape, half, wells, g, harmonic=0.5):
    """harmonic |x|^2 minus Gaussian wells on (-half, half)^d, x fastest (FP64)."""
    d = len(shape)
    xs = [-half + (torch.arange(m, device=DEV, dtype=torch.float64) + 1.0) * (2.0 * half / (m + 1)) for m in shape]
    grid = torch.meshgrid(*xs[::-1], indexing="ij")[::-1]
    u = torch.rand(max(wells, 1), d + 2, generator=g, device=DEV, dtype=torch.float64)
    V = harmonic * sum(x * x for x in grid)
    for k in range(wells):
        r2 = sum((grid[a] - (2.0 * u[k, a] - 1.0) * half) ** 2 for a in range(d))
        V = V - (1.0 + 4.0 * u[k, d]) * torch.exp(-r2 / (2.0 * (0.5 + u[k, d + 1]) ** 2))
    return V.reshape(-1).contiguous()


def _problem(case, g):
    shape = _shape(case)
    half = case["box"]
    V = _potential(shape, half, case["wells"], g, 0.5 if half > 1.0 else 0.0)
    return shape, (-half,) * len(shape), (half,) * len(shape), V


def _randn(n, m, g, dtype=torch.float64):
    return torch.randn(n, m, generator=g, device=DEV, dtype=dtype)


def _padded(X, ld):
    out = torch.zeros(X.shape[0], ld, device=DEV, dtype=X.dtype)
    out[:, : X.shape[1]] = X
    return out


def _ld(p):
    return (p + 7) // 8 * 8


def _orthonormal(n, p, g):
    X = _randn(n, p, g)
    R = torch.linalg.cholesky(X.T @ X).T
    return torch.linalg.solve_triangular(R, X, upper=True, left=False)


def _batch_problems(case, seed):
    g = _gen(seed)
    # sizes belong to the case, values to the seed
    sizes = torch.rand(case["count"], 3, generator=torch.Generator().manual_seed(case["count"]), dtype=torch.float64)
    out = []
    for a, b, w in sizes.tolist():
        N = case["nmin"] + int(a * (case["nmax"] - case["nmin"] + 1))
        p = case["pmin"] + int(b * (case["pmax"] - case["pmin"] + 1))
        V = _potential((N,) * 3, 8.0, 2 + int(10 * w), g)
        out.append(((N,) * 3, (-8.0,) * 3, (8.0,) * 3, V, _randn(N**3, p, g), p))
    return out


def _net_inputs(case, seed):
    g = _gen(seed)
    N, p = case["N"], case["p"]
    V = _potential((N,) * 3, 8.0, 10, g, 0.0)
    c0, c1, c2 = case["c0"], case["c1"], case["c2"]
    layers = [(27, 4, c0), (27, c0, c0), (27, c0, c1), (27, c1, c1), (27, c1, c2), (27, c2, c2), (27, c2 + c1, c1),
              (27, c1, c1), (27, c1 + c0, c1), (27, c1, c1), (1, c1, p)]
    theta = []
    for taps, cin, cout in layers:
        a = math.sqrt(6.0 / (taps * cin))
        theta.append(a * (2.0 * torch.rand(taps * cin * cout, generator=g, device=DEV, dtype=torch.float32) - 1.0))
        theta.append(0.05 * torch.randn(cout, generator=g, device=DEV, dtype=torch.float32))
    return V, torch.cat(theta), layers, g


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return {"case": case, "problems": _batch_problems(case, seed)}
    if kind in ("forward", "gradient"):
        V, theta, _, g = _net_inputs(case, seed)
        net = gb.Net(case["N"], (-8.0,) * 3, (8.0,) * 3, case["p"], (case["c0"], case["c1"], case["c2"]))
        net.set_params(theta.cpu().numpy())
        s = {"case": case, "V": V, "net": net}
        if kind == "gradient":
            s["Ustar"] = _orthonormal(case["N"] ** 3, case["p"], g).float().contiguous()
        return s
    g = _gen(seed)
    p = case["p"]
    if kind == "solve":
        shape, lo, hi, V = _problem(case, g)
        return {"case": case, "args": (shape, lo, hi, V, _randn(V.numel(), p, g), p)}
    if kind == "cg":
        dt = torch.float64 if case["prec"] == "fp64" else torch.float32
        shape, lo, hi, V = _problem(case, g)
        return {"case": case, "geom": (shape, lo, hi), "V": V.to(dt), "sigma": _sigma(shape, lo, hi, V),
                "U": _padded(_orthonormal(V.numel(), p, g).to(dt), _ld(p))}
    n = case["n"]
    if kind == "midpoint":
        U = _orthonormal(n, p, g)
        W = 0.4 * U + 0.2 * _randn(n, p, g) / math.sqrt(n)
        return {"case": case, "U": _padded(U.float(), _ld(p)), "W": _padded(W.float(), _ld(p)), "tau": 1.5}
    U = _randn(n, p, g).div_(math.sqrt(n))
    W = _randn(n, p, g).mul_(0.2 / math.sqrt(n)).add_(U, alpha=0.4)
    s = {"case": case, "U": _padded(U, _ld(p)) if _ld(p) != p else U, "W": _padded(W, _ld(p)) if _ld(p) != p else W}
    if kind == "update64":
        K = 0.02 * _randn(2 * p, p, g) / math.sqrt(p)
        s["KU"] = torch.zeros(_ld(p), _ld(p), device=DEV, dtype=torch.float64)
        s["KU"][:p, :p] = 0.9 * torch.eye(p, device=DEV, dtype=torch.float64) + K[:p]
        s["KW"] = torch.zeros_like(s["KU"])
        s["KW"][:p, :p] = 0.8 * torch.eye(p, device=DEV, dtype=torch.float64) + K[p:]
    return s


# ---- one pass ---------------------------------------------------------------------------
def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind == "solve":
        dt = torch.float64 if c["prec"] == "fp64" else torch.float32
        with gb.Solver(*s["args"], prec=c["prec"], cg_rtol=c["cg_rtol"], device=True) as sol:
            st = sol.step(c["steps"])
            return {"U": sol.get_U_device(dt), "energy": st["energy"]}
    if kind == "batch":
        sols = [gb.Solver(*a, prec="fp32", cg_rtol=c["cg_rtol"], device=True) for a in s["problems"]]
        try:
            with gb.Batch(sols) as b:
                b.step(c["steps"])
            return [{"U": x.get_U_device(torch.float32), "energy": x.stats()["energy"]} for x in sols]
        finally:
            for x in sols:
                x.close()
    if kind == "cg":
        W = torch.zeros_like(s["U"])
        gb.cg_solve(*s["geom"], s["V"], s["sigma"], s["U"], W, c["p"], c["rtol"], precond=c["precond"])
        return W
    if kind == "midpoint":
        p = c["p"]
        C, S, _ = gb.gram(s["U"], s["W"], p)
        _, _, KU, KW = gb.core(C, S, p, s["tau"], dtype=torch.float32)
        return {"U": gb.update(s["U"], s["W"], KU, KW, p), "KU": KU, "KW": KW}
    if kind == "gram64":
        return gb.gram_fp64tc(s["U"], s["W"], c["p"])
    if kind == "update64":
        return gb.update_fp64tc(s["U"], s["W"], s["KU"], s["KW"], c["p"])
    if kind == "forward":
        return s["net"].forward(s["V"])
    return s["net"].loss_grad(s["V"], s["Ustar"], LOSS_WEIGHT)


def work(case):
    """One pass's unavoidable bytes and flops: inputs read once, outputs written once; a solve
    reads and writes U and its warm start W once per step, and takes at least one operator
    application per step."""
    kind = case["kind"]
    if kind == "solve":
        n, p, s = case["nx"] * case["ny"] * case["nz"], case["p"], 8 if case["prec"] == "fp64" else 4
        k = case["steps"]
        return {"bytes": 8.0 * n * (p + 1) + k * 4.0 * n * p * s, "flops": k * n * p * (8.0 * p + 15.0) + 4.0 * n * p * p}
    if kind == "batch":
        sizes = torch.rand(case["count"], 3, generator=torch.Generator().manual_seed(case["count"]), dtype=torch.float64)
        w = {"bytes": 0.0, "flops": 0.0}
        for a, b, _ in sizes.tolist():
            n = (case["nmin"] + int(a * (case["nmax"] - case["nmin"] + 1))) ** 3
            p = case["pmin"] + int(b * (case["pmax"] - case["pmin"] + 1))
            w["bytes"] += 8.0 * n * (p + 1) + case["steps"] * 16.0 * n * p
            w["flops"] += case["steps"] * n * p * (8.0 * p + 15.0) + 4.0 * n * p * p
        return w
    if kind == "cg":
        n, p, s = case["nx"] * case["ny"] * case["nz"], case["p"], 8 if case["prec"] == "fp64" else 4
        return {"bytes": float(n) * s * (3 * p + 1), "flops": 25.0 * n * p}
    if kind in ("midpoint", "gram64", "update64"):
        n, p = float(case["n"]), case["p"]
        if kind == "midpoint":
            return {"bytes": 12.0 * n * p, "flops": 8.0 * n * p * p + 6.0 * p**3}
        if kind == "gram64":
            return {"bytes": 16.0 * n * p + 24.0 * p * p, "flops": 4.0 * n * p * p}
        return {"bytes": 24.0 * n * p + 16.0 * p * p, "flops": 4.0 * n * p * p}
    n, c0, c1, c2, p = float(case["N"]) ** 3, case["c0"], case["c1"], case["c2"], case["p"]
    fine = 27 * (4 * c0 + c0 * c0 + (c1 + c0) * c1 + c1 * c1) + c1 * p
    mid = 27 * (c0 * c1 + c1 * c1 + (c2 + c1) * c1 + c1 * c1)
    low = 27 * (c1 * c2 + c2 * c2)
    f = 2.0 * n * (fine + mid / 8.0 + low / 64.0)
    theta = 4.0 * (fine + mid + low)
    if kind == "forward":
        return {"bytes": n * (8 + 4 * p) + theta, "flops": f}
    return {"bytes": n * (8 + 4 * p) + 2 * theta, "flops": 3.0 * f + 8.0 * n * p * p}


# ---- the same in 64 bits ----------------------------------------------------------------
def _sigma(shape, lo, hi, V):
    return max(0.0, 1.0 - _lowest(shape, lo, hi, V))


def _lowest(shape, lo, hi, V):
    """Lower bound of the spectrum: the discrete Laplacian's lowest level plus min V."""
    low = float(V.min())
    for m, a, b in zip(shape, lo, hi):
        h = (b - a) / (m + 1)
        low += 2.0 / (h * h) * math.sin(math.pi / (2.0 * (m + 1))) ** 2
    return low


class _Operator:
    """H + sigma on n x p blocks, in 64 bits."""

    def __init__(self, shape, lo, hi, V, sigma):
        self.dims = tuple(shape[::-1])
        self.c = [0.5 / ((b - a) / (m + 1)) ** 2 for m, a, b in zip(shape, lo, hi)][::-1]
        self.diag = (V.double() + 2.0 * sum(self.c) + sigma).reshape(*self.dims, 1)

    def __call__(self, X):
        X = X.reshape(*self.dims, -1)
        Y = self.diag * X
        for a, c in enumerate(self.c):
            m = self.dims[a]
            if m > 1:
                Y.narrow(a, 1, m - 1).sub_(X.narrow(a, 0, m - 1), alpha=c)
                Y.narrow(a, 0, m - 1).sub_(X.narrow(a, 1, m - 1), alpha=c)
        return Y.reshape(-1, X.shape[-1])

    def solve(self, U, W):
        """W = (H + sigma)^-1 U by Jacobi-preconditioned CG from W."""
        d = self.diag.reshape(-1, 1)
        R = U - self(W)
        Z = R / d
        P = Z.clone()
        rz = (R * Z).sum(0)
        stop = (1e-13 * U.norm(dim=0)).clamp_min(1e-300)
        for _ in range(4000):
            if bool((R.norm(dim=0) <= stop).all()):
                break
            Q = self(P)
            pq = (P * Q).sum(0)
            a = torch.where(pq > 0, rz / pq, torch.zeros_like(pq))
            W = W + a * P
            R = R - a * Q
            Z = R / d
            new = (R * Z).sum(0)
            P = Z + torch.where(rz > 0, new / rz, torch.zeros_like(rz)) * P
            rz = new
        return W


def _steps(args, steps):
    shape, lo, hi, V, U0, _ = args
    low = _lowest(shape, lo, hi, V)
    sigma = max(0.0, 1.0 - low)
    tau = 1.5 * (low + sigma)
    A = _Operator(shape, lo, hi, V, sigma)
    R = torch.linalg.cholesky(U0.T @ U0).T
    U = torch.linalg.solve_triangular(R, U0, upper=True, left=False)
    W = torch.zeros_like(U)
    for _ in range(steps):
        W = A.solve(U, W)
        KU, KW = _core(W.T @ U, W.T @ W, tau)
        U = U @ KU + W @ KW
    return {"U": U, "energy": 0.5 * float((U * _Operator(shape, lo, hi, V, 0.0)(U)).sum())}


def _core(C, S, tau):
    I = torch.eye(C.shape[0], device=DEV, dtype=torch.float64)
    B = torch.linalg.inv(I + 0.5 * tau * (C - C.T) + 0.25 * tau * tau * (S - C @ C.T))
    return 2.0 * B - I - tau * C.T @ B, tau * B


def _net64(case, theta, layers, V):
    """The network in 64 bits; returns Y and the list of leaf parameters."""
    F = torch.nn.functional
    N = case["N"]
    leaves, at = [], 0
    for taps, cin, cout in layers:
        for m in (taps * cin * cout, cout):
            leaves.append(theta[at:at + m].double().requires_grad_(True))
            at += m

    def conv(i, X):  # X: [channels][z][y][x]
        taps, cin, cout = layers[i]
        if taps == 1:
            return torch.einsum("czyx,co->ozyx", X, leaves[2 * i].reshape(cin, cout)) + leaves[2 * i + 1][:, None, None, None]
        Wt = leaves[2 * i].reshape(3, 3, 3, cin, cout)
        m = X.shape[-1]
        Xp = F.pad(X, (1, 1, 1, 1, 1, 1))
        Z = leaves[2 * i + 1][:, None].expand(cout, m**3)
        for dz in range(3):
            for dy in range(3):
                for dx in range(3):
                    Z = Z + Wt[dz, dy, dx].T @ Xp[:, dz:dz + m, dy:dy + m, dx:dx + m].reshape(cin, m**3)
        return F.silu(Z).reshape(cout, m, m, m)

    def up(X):
        return X.repeat_interleave(2, 1).repeat_interleave(2, 2).repeat_interleave(2, 3)

    x = 2.0 * (torch.arange(N, device=DEV, dtype=torch.float64) + 1.0) / (N + 1) - 1.0
    z, y, xx = torch.meshgrid(x, x, x, indexing="ij")
    X0 = torch.stack([V.reshape(N, N, N) / 6.0, xx, y, z])
    e0 = conv(1, conv(0, X0))
    e1 = conv(3, conv(2, F.avg_pool3d(e0[None], 2)[0]))
    b2 = conv(5, conv(4, F.avg_pool3d(e1[None], 2)[0]))
    d1 = conv(7, conv(6, torch.cat([up(b2), e1])))
    d0 = conv(9, conv(8, torch.cat([up(d1), e0])))
    return conv(10, d0).reshape(case["p"], -1).T, leaves


def exact(case, seed):
    kind = case["kind"]
    if kind == "solve":
        return _steps(prepare(case, seed)["args"], case["steps"])
    if kind == "batch":
        return [_steps(a, case["steps"]) for a in _batch_problems(case, seed)]
    if kind in ("forward", "gradient"):
        V, theta, layers, g = _net_inputs(case, seed)
        with torch.set_grad_enabled(kind == "gradient"):
            Y, leaves = _net64(case, theta, layers, V)
            if kind == "forward":
                return Y
            p = case["p"]
            Us = _orthonormal(case["N"] ** 3, p, g).float().double()
            G, P = Y.T @ Y, Us.T @ Y
            b = torch.trace(G)
            I = torch.eye(p, device=DEV, dtype=torch.float64)
            loss = 1.0 - (P * P).sum() / b + LOSS_WEIGHT * ((p * G / b - I) ** 2).sum() / p**2
            grad = torch.autograd.grad(loss, leaves)
        return float(loss.detach()), np.concatenate([x.cpu().numpy() for x in grad])
    s = prepare(case, seed)
    if kind == "cg":
        shape, lo, hi = s["geom"]
        U = s["U"].double()
        return _Operator(shape, lo, hi, s["V"], s["sigma"]).solve(U, torch.zeros_like(U))
    U, W, ld = s["U"].double(), s["W"].double(), _ld(case["p"])
    if kind == "gram64":
        return W.T @ U, W.T @ W, U.T @ U
    if kind == "update64":
        return U @ s["KU"] + W @ s["KW"]
    p = case["p"]
    KU, KW = _core((W.T @ U)[:p, :p], (W.T @ W)[:p, :p], s["tau"])
    pad = [torch.zeros(ld, ld, device=DEV, dtype=torch.float64) for _ in range(2)]
    pad[0][:p, :p], pad[1][:p, :p] = KU, KW
    return {"U": U @ pad[0] + W @ pad[1], "KU": pad[0], "KW": pad[1]}
