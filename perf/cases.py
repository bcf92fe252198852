"""Performance cases: what a program that uses the solver has it do.

A case names a public entry point (``path``), a vertex grid, the conductivity
field's block size and contrast (log10 k ~ U[-amp, amp] per block of cells)
and the solver's options.  The grids are those of the repository's workloads
and tests (33^3, 65^3, 129^3, 257^3, 513^3) and a ragged one.

``exact`` is a separate float64 restatement in plain torch: the operator, the
V-cycle and a multigrid-preconditioned CG iterated far below the case's
tolerance.  It shares no code with the package.
"""
from __future__ import annotations

import math

import torch
import torch.nn.functional as F

from paper_1604_07163_gb300 import MGSolver, Params, mg_solve

DEV = "cuda"


def _case(name, path, dims, **kw):
    c = dict(name=name, path=path, nz=dims[0], ny=dims[1], nx=dims[2], block=16, amp=2.0, precision="fp64",
             coarse_op="rediscretised", method="cg", face_rule=0, rtol=1e-8)
    c.update(kw)
    return c


def listed():
    return [
        # one operator product of a caller's own Krylov or time-stepping loop on a small grid: launches count
        _case("apply_65", "apply", (65, 65, 65)),
        # the same product at the benchmark grid: memory traffic counts
        _case("apply_257", "apply", (257, 257, 257)),
        # one V-cycle as the preconditioner of a caller's own Krylov method
        _case("vcycle_129", "vcycle", (129, 129, 129)),
        # the smallest whole solve: 33^3, everything in float64, to 1e-10; latency and launches count
        _case("solve_33_fp64", "solve", (33, 33, 33), block=8, amp=1.0, rtol=1e-10),
        # bfloat16 coefficients with Galerkin coarse operators, at a contrast of 10^6
        _case("solve_65_galerkin_bf16k", "solve", (65, 65, 65), block=8, amp=3.0, precision="mixed_bf16k",
              coarse_op="galerkin", rtol=1e-10),
        # a box that is not a cube and not a power of two: ragged tiles on every level, a coarsest level of 120 unknowns
        _case("solve_ragged", "solve", (113, 81, 97), amp=1.0, precision="mixed_fp32", face_rule=1, rtol=1e-10),
        # one step of an inverse problem: hierarchy for a new k, forward solve, loss, adjoint solve, both gradients
        _case("gradient_step_129", "gradient", (129, 129, 129), block=8, amp=1.0, precision="mixed_fp32", rtol=1e-10),
        # the benchmark workload: 257^3, contrast 10^4, float32 V-cycle in float64 CG
        _case("solve_257", "solve", (257, 257, 257), precision="mixed_fp32"),
        # the same solve with every step in float64
        _case("solve_257_fp64", "solve", (257, 257, 257)),
        # the same problem with Galerkin coarse operators
        _case("solve_257_galerkin", "solve", (257, 257, 257), precision="mixed_fp32", coarse_op="galerkin"),
        # the solver of the paper's Sec. 5: flexible GMRES, Galerkin, Richardson(8)-Jacobi, inexact coarsest GMRES
        _case("solve_257_fgmres", "solve", (257, 257, 257), precision="mixed_fp32", coarse_op="galerkin",
              method="fgmres_richardson8"),
        # the large workload: 513^3, contrast 10^6, Galerkin coarse operators
        _case("solve_513_galerkin", "solve", (513, 513, 513), amp=3.0, precision="mixed_fp32", coarse_op="galerkin"),
    ]


def draw(rng):
    """One more case of the same paths: 17 to 289 vertices per axis (spread over the logarithm), each axis of its
    own, a multiple of 2^m intervals so that the grid coarsens m times."""
    path = rng.choice(["apply", "vcycle", "solve", "solve", "solve", "gradient"])
    m = rng.choice([2, 3, 3, 4])
    top = 160 if path == "gradient" else 288
    size = math.exp(rng.uniform(math.log(16), math.log(top)))

    def axis():
        cells = size * rng.choice([0.75, 1.0, 1.0, 1.25])
        # 3 to 7 cells at the end of the coarsening at most for the coarser grids, more halvings for the finer ones
        h = 2 ** max(m, math.ceil(math.log2(max(cells, 1) / 7.0)))
        return min(top, max(4, round(cells / h)) * h) + 1

    dims = tuple(axis() for _ in range(3))
    c = _case("", path, dims, block=rng.choice([4, 8, 16]), amp=rng.choice([0.5, 1.0, 1.5]), rtol=1e-10)
    del c["name"]
    if path == "solve":
        c["precision"] = rng.choice(["fp64", "mixed_fp32", "mixed_fp32", "mixed_bf16k"])
        c["coarse_op"] = rng.choice(["rediscretised", "galerkin"])
        c["face_rule"] = rng.choice([0, 1])
        if c["coarse_op"] == "galerkin":
            c["amp"] = rng.choice([1.0, 2.0, 3.0])
            c["method"] = rng.choice(["cg", "cg", "fgmres_richardson8"])
    elif path == "gradient":
        c["precision"] = rng.choice(["fp64", "mixed_fp32"])
        c["amp"] = 1.0
        c["face_rule"] = rng.choice([0, 1])
    return c


def _dims(case):
    return case["nz"], case["ny"], case["nx"]


def _log_k(case, seed):
    """ln k per cell: one value per block of cells."""
    g = torch.Generator(device=DEV).manual_seed(2 * seed + 1)
    cells = [n - 1 for n in _dims(case)]
    b = case["block"]
    u = torch.rand([-(-n // b) for n in cells], dtype=torch.float64, device=DEV, generator=g)
    v = (2 * u - 1) * (case["amp"] * math.log(10.0))
    for a in range(3):
        v = v.repeat_interleave(b, dim=a).narrow(a, 0, cells[a])
    return v.contiguous()


def _nodal(case, seed):
    """U[-1, 1] at interior nodes, 0 on the boundary."""
    g = torch.Generator(device=DEV).manual_seed(2 * seed + 2)
    v = torch.rand(_dims(case), dtype=torch.float64, device=DEV, generator=g).mul_(2).sub_(1)
    out = torch.zeros_like(v)
    out[1:-1, 1:-1, 1:-1] = v[1:-1, 1:-1, 1:-1]
    return out


def _observations(case, seed):
    """Mask of the observed nodes (5 % of the interior) and the observed values."""
    g = torch.Generator(device=DEV).manual_seed(2 * seed + 2000003)
    mask = (torch.rand(_dims(case), dtype=torch.float64, device=DEV, generator=g) < 0.05).to(torch.float64)
    obs = torch.rand(_dims(case), dtype=torch.float64, device=DEV, generator=g).mul_(2).sub_(1).mul_(1e-3)
    return mask, obs


def _params(case):
    p = dict(precision=case["precision"], coarse_op=case["coarse_op"], face_rule=case["face_rule"])
    if case["method"] == "fgmres_richardson8":
        p.update(krylov="fgmres", smoother="richardson", nu_pre=8, nu_post=8)
        # the inexact coarsest solve needs a coarsest level of at most 32 unknowns
        if _coarsest(_dims(case)) <= 32:
            p.update(coarse_solve="gmres")
    return Params(**p)


def _coarsest(dims):
    d = list(dims)
    while all((n - 1) % 2 == 0 and (n - 1) // 2 + 1 >= 5 for n in d):
        d = [(n - 1) // 2 + 1 for n in d]
    return (d[0] - 2) * (d[1] - 2) * (d[2] - 2)


def prepare(case, seed):
    """Inputs, and for all but the gradient step the hierarchy a program keeps for its k."""
    s = {"case": case, "logk": _log_k(case, seed), "f": _nodal(case, seed), "params": _params(case)}
    if case["path"] == "gradient":
        s["mask"], s["obs"] = _observations(case, seed)
        s["logk"].requires_grad_(True)
        s["f"].requires_grad_(True)
    else:
        s["solver"] = MGSolver(s.pop("logk"), s["params"], k_is_log=True)
    return s


def run(state):
    case = state["case"]
    if case["path"] == "apply":
        return state["solver"].apply(state["f"], -1)
    if case["path"] == "vcycle":
        return state["solver"].vcycle(state["f"])
    if case["path"] == "solve":
        return state["solver"].solve(state["f"], case["rtol"])[0]
    phi = mg_solve(state["f"], state["logk"], state["params"], case["rtol"])
    loss = 0.5 * (state["mask"] * (phi - state["obs"]) ** 2).sum()
    grad_f, grad_logk = torch.autograd.grad(loss, (state["f"], state["logk"]))
    return {"phi": phi.detach(), "grad_f": grad_f, "grad_logk": grad_logk}


def work(case):
    """Inputs read once, outputs written once; the flops of one operator product on them."""
    nodes = case["nz"] * case["ny"] * case["nx"]
    arrays = {"apply": 3, "vcycle": 3, "solve": 3, "gradient": 7}[case["path"]]
    return {"bytes": 8.0 * arrays * nodes, "flops": 13.0 * nodes}


# ------------------------------------------------------------------ exact
def _edges(k, face_rule):
    """h_a^-2 times the mean of the four cells around each edge, per axis (z, y, x)."""
    out = []
    for a in range(3):
        p, q = [d for d in range(3) if d != a]
        v = k if face_rule else 1.0 / k
        s = v
        for d in (p, q):
            n = s.shape[d] - 1
            s = s.narrow(d, 0, n) + s.narrow(d, 1, n)
        out.append((0.25 * s if face_rule else 4.0 / s) * float(k.shape[a]) ** 2)
    return out


class _Level:
    def __init__(self, k, face_rule):
        self.c = _edges(k, face_rule)
        self.shape = tuple(n - 1 for n in k.shape)
        self.diag = sum(c.narrow(a, 0, self.shape[a]) + c.narrow(a, 1, self.shape[a]) for a, c in enumerate(self.c))

    def apply(self, u):
        y = self.diag * u
        for a, c in enumerate(self.c):
            n = self.shape[a]
            y.narrow(a, 1, n - 1).sub_(c.narrow(a, 1, n - 1) * u.narrow(a, 0, n - 1))
            y.narrow(a, 0, n - 1).sub_(c.narrow(a, 1, n - 1) * u.narrow(a, 1, n - 1))
        return y


def _restrict(r):
    for a in range(3):
        n = (r.shape[a] - 1) // 2
        i = 2 * torch.arange(n, device=r.device)
        r = 0.25 * (r.index_select(a, i) + r.index_select(a, i + 2)) + 0.5 * r.index_select(a, i + 1)
    return r


def _prolong(e):
    for a in range(3):
        pad = [0, 0, 0, 0, 0, 0]
        pad[2 * (2 - a)] = pad[2 * (2 - a) + 1] = 1
        g = F.pad(e, pad)
        n = e.shape[a]
        i = torch.arange(2 * n + 1, device=e.device)
        e = 0.5 * (g.index_select(a, (i + 1) // 2) + g.index_select(a, i // 2 + 1))
    return e


class _Multigrid:
    """V(2,2), Chebyshev(2)-Jacobi on [0.2, 2], re-discretised coarse operators, dense coarsest solve."""

    def __init__(self, k, face_rule):
        self.lv = [_Level(k, face_rule)]
        while all(n % 2 == 0 and n // 2 + 1 >= 5 for n in k.shape):
            k = F.avg_pool3d(k[None, None], 2)[0, 0]
            self.lv.append(_Level(k, face_rule))
        c = self.lv[-1]
        n = c.shape[0] * c.shape[1] * c.shape[2]
        eye = torch.eye(n, dtype=torch.float64, device=k.device)
        self.coarse = torch.linalg.cholesky(
            torch.stack([c.apply(eye[i].reshape(c.shape)).reshape(-1) for i in range(n)], 1))

    def smooth(self, lv, b, x):
        alpha, beta = 0.2, 2.0
        theta, delta = 0.5 * (alpha + beta), 0.5 * (beta - alpha)
        sigma = theta / delta
        s = b / lv.diag if x is None else (b - lv.apply(x)) / lv.diag
        d = s / theta
        x = d if x is None else x + d
        rho = 1.0 / (2.0 * sigma - 1.0 / sigma)
        d = rho / sigma * d + 2.0 * rho / delta * ((b - lv.apply(x)) / lv.diag)
        return x + d

    def vcycle(self, b, l=0):
        lv = self.lv[l]
        if l + 1 == len(self.lv):
            return torch.cholesky_solve(b.reshape(-1, 1), self.coarse).reshape(lv.shape)
        x = self.smooth(lv, b, None)
        x = x + _prolong(self.vcycle(_restrict(b - lv.apply(x)), l + 1))
        return self.smooth(lv, b, x)

    def solve(self, f, rtol=1e-13, maxit=400):
        """CG until the residual is below rtol or stops falling; the iterate of the smallest residual."""
        x, r = torch.zeros_like(f), f.clone()
        p, rho, best, keep = None, 1.0, math.inf, x
        bnorm = float(f.norm())
        for it in range(maxit):
            z = self.vcycle(r)
            new = torch.sum(r * z)
            p = z if p is None else z + (new / rho) * p
            rho = new
            q = self.lv[0].apply(p)
            a = rho / torch.sum(p * q)
            x, r = x + a * p, r - a * q
            if it % 5 == 4:
                r = f - self.lv[0].apply(x)  # the true residual
                res = float(r.norm()) / bnorm
                if res < best:
                    best, keep = res, x
                if res <= rtol or res > 100 * best:
                    break
        return keep


def _inner(v):
    return v[1:-1, 1:-1, 1:-1].contiguous()


def _outer(v):
    return F.pad(v, [1, 1, 1, 1, 1, 1])


def _gradient(k, face_rule, edges, phi, lam):
    """dL/dln k per cell: every edge's -h^-2 dlam dphi dk_e/dln k_c, added to its four cells."""
    g = torch.zeros_like(k)
    for a in range(3):
        p, q = [d for d in range(3) if d != a]
        t = -torch.diff(phi, dim=a) * torch.diff(lam, dim=a)
        for d in (p, q):
            t = t.narrow(d, 1, t.shape[d] - 2)
        ih2 = float(k.shape[a]) ** 2
        t = t * (0.25 * ih2 if face_rule else edges[a] ** 2 / (4.0 * ih2))
        for i in (0, 1):
            for j in (0, 1):
                view = g.narrow(p, i, g.shape[p] - 1).narrow(q, j, g.shape[q] - 1)
                view.add_(t)
    return g * k if face_rule else g / k


def exact(case, seed):
    nodes = case["nz"] * case["ny"] * case["nx"]
    hard = case["path"] in ("solve", "gradient") and (case["amp"] > 1.0 or case["coarse_op"] == "galerkin")
    if nodes > (1 << 21) * 1.1 and (hard or nodes > 1 << 24) and case["path"] != "apply":
        return None
    with torch.no_grad():
        k, f = torch.exp(_log_k(case, seed)), _inner(_nodal(case, seed))
        if case["path"] == "apply":
            return _outer(_Level(k, case["face_rule"]).apply(f))
        m = _Multigrid(k, case["face_rule"])
        if case["path"] == "vcycle":
            return _outer(m.vcycle(f))
        if case["path"] == "solve":
            return _outer(m.solve(f))
        mask, obs = _observations(case, seed)
        phi = m.solve(f)
        g = _outer(_inner(mask) * (phi - _inner(obs)))
        lam = _outer(m.solve(_inner(g)))
        phi = _outer(phi)
        return {"phi": phi, "grad_f": lam, "grad_logk": _gradient(k, case["face_rule"], m.lv[0].c, phi, lam)}
