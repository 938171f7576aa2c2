"""The measured work of the library: what a user has it do through its Python entry points.

Every case is a finite-element system on a structured grid of the unit cube (trilinear
hexahedra, Dirichlet boundary) with its octree of sub-domains, as the library's own grid
builders make them; values and loads come from the seed.  The kinds of work:

  solve      RSD.setup and RSD.solve: one system, one right-hand side, handle released
  resolve    RSD.solve on a hierarchy that the program keeps (a sequence of loads)
  apply      RSD.apply on a kept hierarchy (a program with its own Krylov loop)
  gradient   diffusion_solve forward and backward: u, dL/dm and dL/db
  batched    RSD.setup_batched and RSD.solve for many independent problems
  elastic    as solve, for 3-D linear elasticity (three unknowns per node)
  paper      as solve, in the paper's own mode (V-hat truncation, gamma inner iterations)
  convection as solve, for a nonsymmetric convection-diffusion system (LU fronts)

Solves run to a relative residual of 1e-12, the tolerance of the paper's experiments.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1210_6266_gb300 as rsd

TOL = 1e-12
PREC = {"fp64": rsd.RSD_PREC_FP64, "fp32": rsd.RSD_PREC_FP32, "tf32": rsd.RSD_PREC_TF32,
        "fp16": rsd.RSD_PREC_FP16, "bf16": rsd.RSD_PREC_BF16}
POISSON_RATIO = 0.3


# ---- the cases --------------------------------------------------------------------------

def listed() -> list[dict]:
    return [
        # the smallest system of the configurations (13^3 nodes, 8 sub-domains, FP64): a call
        # made inside another program's loop, where launches and host work are all there is
        dict(name="solve13_fp64", kind="solve", n=13, depth=1, prec="fp64"),
        # an interactive-size system with RSD.setup's default precisions (TF32 sub-domains,
        # FP64 root), odd box sizes on every level
        dict(name="solve38_default", kind="solve", n=38, depth=2, prec="default"),
        # the plain FP64 form that the mixed forms are judged against, one PCG iteration
        dict(name="solve57_fp64", kind="solve", n=57, depth=2, prec="fp64"),
        # the headline: 129^3 log-normal diffusion, 512 sub-domains, FP16 operand copies
        dict(name="solve129_fp16", kind="solve", n=129, depth=3, prec="fp16"),
        # one hierarchy, a sequence of loads (time steps, many sources), TF32 factors
        dict(name="resolve97_tf32", kind="resolve", n=97, depth=3, prec="tf32"),
        # the preconditioner inside a caller's own iteration, FP64 factors
        dict(name="apply49_fp64", kind="apply", n=49, depth=2, prec="fp64"),
        # inverse problems: value and gradients with diffusion_solve's defaults (all FP64)
        dict(name="gradient33_fp64", kind="gradient", n=33, depth=2, prec="fp64"),
        # and the 65^3 configuration of that workload in its mixed form
        dict(name="gradient65_tf32", kind="gradient", n=65, depth=2, prec="tf32"),
        # many independent Poisson problems of uneven size in one hierarchy, BF16 operands
        dict(name="batched24_bf16", kind="batched", count=24, lo=17, hi=65, prec="bf16"),
        # linear elasticity, sub-domain moduli over three decades
        dict(name="elastic49_tf32", kind="elastic", n=49, depth=3, prec="tf32"),
        # the paper's Algorithm 2 with eight inner GMRES iterations, FGMRES outside
        dict(name="paper65_gamma8", kind="paper", n=65, depth=3, prec="fp16", gamma=8),
        # nonsymmetric fronts: convection-diffusion, LU in FP64
        dict(name="convection37_fp64", kind="convection", n=37, depth=2, prec="fp64"),
    ]


def _depth(n: int) -> int:
    """Sub-domains of about 7 to 16 nodes a side."""
    return max(1, min(3, round(math.log2(max(n - 1, 2) / 12.0))))


def _log_size(rng, lo: int, hi: int) -> int:
    return max(lo, min(hi, round(lo * (hi / lo) ** rng.random())))


def draw(rng) -> dict:
    kind = rng.choice(["solve", "solve", "solve", "resolve", "apply", "gradient", "gradient", "batched",
                       "elastic", "paper", "convection"])
    if kind == "solve":
        prec = rng.choice(["fp64", "default", "tf32", "fp16"])
        n = _log_size(rng, 13, {"fp64": 56, "default": 56}.get(prec, 120))
    elif kind == "resolve":
        prec, n = rng.choice(["fp64", "tf32", "fp16"]), 0
        n = _log_size(rng, 17, 56 if prec == "fp64" else 96)
    elif kind == "apply":
        prec, n = "fp64", _log_size(rng, 13, 56)
    elif kind == "gradient":
        prec = rng.choice(["fp64", "fp64", "tf32"])
        n = _log_size(rng, 13, 48 if prec == "fp64" else 72)
    elif kind == "batched":
        lo = rng.randint(13, 24)
        return dict(kind=kind, count=_log_size(rng, 4, 32), lo=lo, hi=rng.randint(lo + 8, 56),
                    prec=rng.choice(["bf16", "tf32"]))
    elif kind == "elastic":
        prec, n = rng.choice(["tf32", "fp16"]), _log_size(rng, 13, 48)
    elif kind == "paper":
        n = _log_size(rng, 21, 64)
        return dict(kind=kind, n=n, depth=_depth(n), prec=rng.choice(["fp16", "tf32", "fp64"]),
                    gamma=rng.choice([4, 8]))
    else:
        prec, n = "fp64", _log_size(rng, 13, 37)
    return dict(kind=kind, n=n, depth=_depth(n), prec=prec)


# ---- inputs -----------------------------------------------------------------------------

def _precs(case) -> dict:
    if case["prec"] == "default":
        return {}
    p = PREC[case["prec"]]
    return dict(prec_leaf=p, prec_mid=p, prec_root=p)


def _scalar_inputs(case, seed: int):
    """Log-normal coefficient per element (sigma = 1) and nodal load in [-1, 1]."""
    n = case["n"]
    g = np.random.default_rng(seed)
    return np.exp(g.standard_normal((n - 1) ** 3)), g.uniform(-1.0, 1.0, (n - 2) ** 3)


def _batched_inputs(case, seed: int):
    """Sizes are part of the case; Poisson problems with loads from the seed."""
    sizes = np.random.default_rng(4).integers(case["lo"], case["hi"] + 1, case["count"])
    g = np.random.default_rng(seed)
    return [(int(n), 1 if n - 1 < 32 else 2, g.uniform(-1.0, 1.0, (int(n) - 2) ** 3)) for n in sizes]


def _elastic_inputs(case, seed: int):
    """Young's modulus per leaf log-uniform in [1, 1e3], load per unknown in [-1, 1]."""
    g = np.random.default_rng(seed)
    return 10.0 ** g.uniform(0.0, 3.0, 8 ** case["depth"]), g.uniform(-1.0, 1.0, 3 * (case["n"] - 2) ** 3)


def _gradient_inputs(case, seed: int):
    """m: a Gaussian field of correlation length 0.1; loads in [-1, 1]; observations: a
    smooth bump of the solution's size."""
    n, ne = case["n"], case["n"] - 1
    g = np.random.default_rng(seed)
    i = np.arange(ne)
    k = np.exp(-0.5 * ((i[:, None] - i[None, :]) / (0.1 * ne)) ** 2)
    z = np.einsum("ai,bj,ck,ijk->abc", k, k, k, g.standard_normal((ne, ne, ne)), optimize=True)
    m = ((z - z.mean()) / z.std()).reshape(-1)
    b = g.uniform(-1.0, 1.0, (n - 2) ** 3) / ne ** 3
    s = np.sin(np.pi * np.arange(1, n - 1) / ne)
    u_obs = (1e-3 * g.uniform(0.5, 1.5) * s[:, None, None] * s[None, :, None] * s[None, None, :]).reshape(-1)
    return m, b, u_obs


def _velocity(seed: int) -> np.ndarray:
    """A constant velocity with element Peclet numbers of order one."""
    return np.random.default_rng(seed + 1).uniform(-20.0, 20.0, 3)


def _add_convection(prob, vel) -> torch.Tensor:
    """Values of K with the (skew) Galerkin matrix of vel . grad added on K's pattern."""
    n, h, m = prob["n"], 1.0 / (prob["n"] - 1), prob["n"] - 2
    rowptr, col = prob["rowptr"], prob["col"].to(torch.int64)
    row = torch.repeat_interleave(torch.arange(prob["n_dof"], device=col.device), rowptr[1:] - rowptr[:-1])
    mass = torch.tensor([h / 6, 4 * h / 6, h / 6], dtype=torch.float64, device=col.device)
    grad = torch.tensor([-0.5, 0.0, 0.5], dtype=torch.float64, device=col.device)
    d = [col % m - row % m + 1, col // m % m - row // m % m + 1, col // (m * m) - row // (m * m) + 1]
    add = torch.zeros_like(prob["val"])
    for a in range(3):
        t = torch.full_like(add, float(vel[a]))
        for c in range(3):
            t = t * (grad if c == a else mass)[d[c]]
        add += t
    return prob["val"] + add


def _setup(prob, case, **kw):
    return rsd.RSD.setup(prob["rowptr"], prob["col"], prob["val"], prob["dof_node"], prob["parent"],
                         **_precs(case), **kw)


def prepare(case: dict, seed: int) -> dict:
    kind = case["kind"]
    if kind == "batched":
        return dict(case=case, probs=(p := [rsd.grid_problem(n, d, np.ones((n - 1) ** 3), f)
                                            for n, d, f in _batched_inputs(case, seed)]),
                    b=torch.cat([q["b"] for q in p]))
    if kind == "gradient":
        m, b, u_obs = (torch.as_tensor(v, device="cuda") for v in _gradient_inputs(case, seed))
        return dict(case=case, m=m, b=b, u_obs=u_obs)
    if kind == "elastic":
        E, f = _elastic_inputs(case, seed)
        return dict(case=case, prob=rsd.grid_problem_elastic(case["n"], case["depth"], E, POISSON_RATIO, f))
    kappa, f = _scalar_inputs(case, seed)
    prob = rsd.grid_problem(case["n"], case["depth"], kappa, f)
    if kind == "convection":
        prob["val"] = _add_convection(prob, _velocity(seed))
    state = dict(case=case, prob=prob)
    if kind in ("resolve", "apply"):
        state["h"] = _setup(prob, case)
    return state


def run(state: dict):
    case = state["case"]
    kind = case["kind"]
    if kind == "apply":
        return state["h"].apply(state["prob"]["b"])
    if kind == "resolve":
        return state["h"].solve(state["prob"]["b"], tol=TOL)[0]
    if kind == "gradient":
        m, b = state["m"].detach().requires_grad_(), state["b"].detach().requires_grad_()
        kw = {} if case["prec"] == "fp64" else dict(tol=TOL, precs=(PREC[case["prec"]],) * 3)
        u = rsd.diffusion_solve(m, b, case["n"], case["depth"], **kw)
        loss = 0.5 * ((u - state["u_obs"]) ** 2).sum()
        dm, db = torch.autograd.grad(loss, (m, b))
        return u.detach(), dm, db
    if kind == "batched":
        h, b = rsd.RSD.setup_batched(state["probs"], **_precs(case)), state["b"]
    else:
        kw = {}
        if kind == "paper":
            kw = dict(mode=rsd.RSD_MODE_PAPER, gamma=case["gamma"], maxit=1000)
        elif kind == "convection":
            kw = dict(nonsymmetric=True)
        h, b = _setup(state["prob"], case, **kw), state["prob"]["b"]
    u, _ = h.solve(b, tol=TOL)
    h.close()
    return u


# ---- the work no implementation can do without --------------------------------------------

def _fronts(n: int, depth: int):
    """(s, b) of every octree node: own unknowns, and ancestors' unknowns around its box."""
    def axis(lo, hi, d):
        if d == 0:
            return [(lo, hi)]
        mid = lo + (hi - lo) // 2
        return axis(lo, mid, d - 1) + axis(mid, hi, d - 1)

    out = []
    for d in range(depth + 1):
        cells = []
        for lo, hi in axis(0, n - 1, d):
            inner = max(hi - lo - 1, 0)
            ext = inner + (lo > 0) + (hi < n - 1)
            below = max(inner - 1, 0) if d < depth else 0
            cells.append((inner, ext, below))
        for x in cells:
            for y in cells:
                for z in cells:
                    vol = x[0] * y[0] * z[0]
                    s = vol - (x[2] * y[2] * z[2] if d < depth else 0)
                    out.append((s, x[1] * y[1] * z[1] - vol))
    return out


def work(case: dict) -> dict:
    if case["kind"] == "batched":
        grids = [(n, d) for n, d, _ in _batched_inputs(case, 0)]
    else:
        grids = [(case["n"], case["depth"])]
    comps = 3 if case["kind"] == "elastic" else 1
    flops = bytes_ = factor = 0.0
    for n, depth in grids:
        dof = comps * (n - 2) ** 3
        nnz = comps * comps * (3 * (n - 2) - 2) ** 3
        fronts = [(comps * s, comps * b) for s, b in _fronts(n, depth)]
        if case["kind"] == "paper":                  # the leaves are the only factored fronts
            fronts = fronts[-8 ** depth:]
        flops += sum(s ** 3 / 3 + s * s * b + s * b * b for s, b in fronts)
        factor += sum(s * s / 2 + s * b for s, b in fronts)
        bytes_ += 12.0 * nnz + 8.0 * dof + 16.0 * dof   # K once, load in, solution out
    if case["kind"] == "convection":
        flops, factor = 2 * flops, 2 * factor
    if case["kind"] in ("apply", "resolve"):
        # the kept factors once; TF32 and FP16 hierarchies are read through 16-bit copies
        return dict(bytes=(8.0 if case["prec"] == "fp64" else 2.0) * factor + bytes_, flops=4.0 * factor)
    if case["kind"] == "gradient":
        bytes_ += 24.0 * (case["n"] - 1) ** 3
    return dict(bytes=bytes_, flops=flops)


# ---- the same answers in 64 bits, from plain torch ------------------------------------------

def _gauss_basis():
    """Gradients of the eight trilinear shape functions at the 2 x 2 x 2 Gauss points."""
    pts = np.array([0.5 - 0.5 / math.sqrt(3.0), 0.5 + 0.5 / math.sqrt(3.0)])
    corner = [(i & 1, i >> 1 & 1, i >> 2 & 1) for i in range(8)]
    val, grad = [], []
    for z in pts:
        for y in pts:
            for x in pts:
                f = [(1 - x, x), (1 - y, y), (1 - z, z)]
                val.append([f[0][a] * f[1][b] * f[2][c] for a, b, c in corner])
                grad.append([[(2 * a - 1) * f[1][b] * f[2][c], f[0][a] * (2 * b - 1) * f[2][c],
                              f[0][a] * f[1][b] * (2 * c - 1)] for a, b, c in corner])
    return np.array(val), np.array(grad)                # (8, 8), (8, 8, 3)


def _laplace_element() -> np.ndarray:
    _, g = _gauss_basis()
    return np.einsum("qad,qbd->ab", g, g) / 8.0


def _elastic_element(nu: float) -> np.ndarray:
    _, g = _gauss_basis()
    lam, mu = nu / ((1 + nu) * (1 - 2 * nu)), 0.5 / (1 + nu)
    eye = np.eye(3)
    k = (lam * np.einsum("qai,qbj->aibj", g, g) + mu * np.einsum("qaj,qbi->aibj", g, g)
         + mu * np.einsum("qad,qbd,ij->aibj", g, g, eye)) / 8.0
    return k.reshape(24, 24)


class _Operator:
    """K x = sum_e G_e^T (coef_e A + B) G_e x by element gathers; x: (n-2)^3 nodes of c
    components, A and B (8c x 8c), coef per element in x-fastest order."""

    def __init__(self, n, coef, A, B=None, comps=1):
        dev = "cuda"
        self.n, self.c = n, comps
        self.coef = torch.as_tensor(coef, dtype=torch.float64, device=dev).reshape(n - 1, n - 1, n - 1)
        self.A = torch.as_tensor(A, dtype=torch.float64, device=dev)
        self.B = None if B is None else torch.as_tensor(B, dtype=torch.float64, device=dev)

    def gather(self, x):
        n, c = self.n, self.c
        full = torch.zeros(n, n, n, c, dtype=torch.float64, device="cuda")
        full[1:-1, 1:-1, 1:-1] = x.reshape(n - 2, n - 2, n - 2, c)
        e = n - 1
        return torch.cat([full[k >> 2 & 1:(k >> 2 & 1) + e, k >> 1 & 1:(k >> 1 & 1) + e, k & 1:(k & 1) + e]
                          for k in range(8)], dim=-1)

    def __call__(self, x):
        n, c, e = self.n, self.c, self.n - 1
        g = self.gather(x)
        y = (g @ self.A.T) * self.coef[..., None]
        if self.B is not None:
            y += g @ self.B.T
        full = torch.zeros(n, n, n, c, dtype=torch.float64, device="cuda")
        for k in range(8):
            full[k >> 2 & 1:(k >> 2 & 1) + e, k >> 1 & 1:(k >> 1 & 1) + e, k & 1:(k & 1) + e] += y[..., k * c:(k + 1) * c]
        return full[1:-1, 1:-1, 1:-1].reshape(-1)

    def diagonal(self):
        n, c, e = self.n, self.c, self.n - 1
        full = torch.zeros(n, n, n, c, dtype=torch.float64, device="cuda")
        for k in range(8):
            d = self.A.diagonal()[k * c:(k + 1) * c]
            full[k >> 2 & 1:(k >> 2 & 1) + e, k >> 1 & 1:(k >> 1 & 1) + e, k & 1:(k & 1) + e] += self.coef[..., None] * d
        return full[1:-1, 1:-1, 1:-1].reshape(-1)


def _cg(op, f, maxit=12000):
    """Jacobi-preconditioned CG, restarted on the true residual until it stops falling."""
    inv, x, best = 1.0 / op.diagonal(), torch.zeros_like(f), None
    fn = f.norm()
    for _ in range(4):
        r = f - op(x)
        rel = float(r.norm() / fn)
        if best is not None and rel > 0.2 * best:
            break
        best = rel
        z = inv * r
        p, rz, r0 = z.clone(), r @ z, r.norm()
        d = torch.zeros_like(f)
        for it in range(maxit):
            q = op(p)
            a = rz / (p @ q)
            d += a * p
            r = r - a * q
            if it % 25 == 24 and float(r.norm() / r0) < 1e-12:
                break
            z = inv * r
            new = r @ z
            p = z + (new / rz) * p
            rz = new
        x = x + d
    return x


def _bicgstab(op, f, maxit=6000):
    """Jacobi-preconditioned BiCGStab, restarted on the true residual."""
    inv, x = 1.0 / op.diagonal(), torch.zeros_like(f)
    fn = f.norm()
    for _ in range(12):
        r = f - op(x)
        if float(r.norm() / fn) < 2e-15:
            break
        r_hat, rho, p, r0 = r.clone(), r @ r, r.clone(), r.norm()
        d = torch.zeros_like(f)
        for it in range(maxit):
            ph = inv * p
            v = op(ph)
            a = rho / (r_hat @ v)
            s = r - a * v
            sh = inv * s
            t = op(sh)
            w = (t @ s) / (t @ t)
            d += a * ph + w * sh
            r = s - w * t
            if it % 10 == 9 and not float(r.norm() / r0) > 1e-9:
                break
            new = r_hat @ r
            p = r + (new / rho) * (a / w) * (p - w * v)
            rho = new
        if not bool(torch.isfinite(d).all()):
            break
        x = x + d
    return x


def _leaf_coefficient(n: int, depth: int, E: np.ndarray) -> np.ndarray:
    """E of the octree leaf of every element (breadth-first leaf order)."""
    lo, hi = np.zeros(n - 1, dtype=int), np.full(n - 1, n - 1)
    e = np.arange(n - 1)
    leaf = np.zeros((n - 1,) * 3, dtype=int)
    for _ in range(depth):
        mid = lo + (hi - lo) // 2
        up = (e >= mid).astype(int)
        lo, hi = np.where(up, mid, lo), np.where(up, hi, mid)
        leaf = 8 * leaf + up[None, None, :] + 2 * up[None, :, None] + 4 * up[:, None, None]
    return E[leaf]


def _convection_element(vel, h: float) -> np.ndarray:
    val, g = _gauss_basis()
    return h * h * np.einsum("qa,qbd,d->ab", val, g, np.asarray(vel)) / 8.0


def exact(case: dict, seed: int):
    kind = case["kind"]
    lap = _laplace_element()
    if kind == "batched":
        out = []
        for n, _, f in _batched_inputs(case, seed):
            h = 1.0 / (n - 1)
            out.append(_cg(_Operator(n, np.full((n - 1) ** 3, h), lap), torch.as_tensor(f * h ** 3, device="cuda")))
        return torch.cat(out)
    n, h = case["n"], 1.0 / (case["n"] - 1)
    if kind == "gradient":
        m, b, u_obs = (torch.as_tensor(v, device="cuda") for v in _gradient_inputs(case, seed))
        kappa = torch.exp(m)
        op = _Operator(n, h * kappa, lap)
        u = _cg(op, b)
        lam = _cg(op, u - u_obs)
        dm = -(op.gather(lam) * (op.gather(u) @ op.A.T)).sum(-1) * op.coef
        return u, dm.reshape(-1), lam
    if kind == "elastic":
        E, f = _elastic_inputs(case, seed)
        op = _Operator(n, h * _leaf_coefficient(n, case["depth"], E), _elastic_element(POISSON_RATIO), comps=3)
        return _cg(op, torch.as_tensor(f * h ** 3, device="cuda"))
    kappa, f = _scalar_inputs(case, seed)
    b = torch.as_tensor(f * h ** 3, device="cuda")
    if kind == "convection":
        return _bicgstab(_Operator(n, h * kappa, lap, _convection_element(_velocity(seed), h)), b)
    return _cg(_Operator(n, h * kappa, lap), b)
