"""Timed cases: what a program that uses the partial-reuse AMG solver has it do.

Every case is one pass of a time-stepping (or optimisation) program through the
public entry points: the values of the step's matrix, the hierarchy refreshed
by the strategy in use, the solve to a relative residual of 1e-8.  The state of
a case is a running series: the pattern is known, the full setup of the first
step is done and one later step has been taken, as in the middle of such a run.

The fields are those of the collapsing water column (density 1000 in the column,
1 in the air): the column's front stands where the seed puts it, and the
right-hand side is drawn from the seed.
"""
from __future__ import annotations

import math

import torch

from paper_2108_02054_gb300 import amg as B
from paper_2108_02054_gb300 import autograd as AD

TOL = 1e-8        # relative residual of the time steps' solves
GRAD_TOL = 1e-10  # and of the differentiable solve (PoissonSolver's default)
STEPS = 100       # the column's front moves through this many positions


def listed():
    return [
        # 32 x 32 cells, FP64: the smallest system of the configurations; one
        # time step is launch and latency time
        {"name": "step_2d32", "kind": "poisson", "dim": 2, "N": 32, "precision": "fp64", "flavour": "sa", "mode": "partial"},
        # an ordinary 2D grid of an odd size
        {"name": "step_2d301", "kind": "poisson", "dim": 2, "N": 301, "precision": "fp64", "flavour": "sa", "mode": "partial"},
        # the 3D FP64 configuration
        {"name": "step_3d64", "kind": "poisson", "dim": 3, "N": 64, "precision": "fp64", "flavour": "sa", "mode": "partial"},
        # the two mixed-precision configurations (FP32 hierarchy, FP64 CG); the
        # second is the largest system of all
        {"name": "step_3d128_mixed", "kind": "poisson", "dim": 3, "N": 128, "precision": "mixed", "flavour": "sa", "mode": "partial"},
        {"name": "step_3d192_mixed", "kind": "poisson", "dim": 3, "N": 192, "precision": "mixed", "flavour": "sa", "mode": "partial"},
        # the paper's own flavour (plain aggregation, damped Jacobi), odd size
        {"name": "plain_3d71", "kind": "poisson", "dim": 3, "N": 71, "precision": "fp64", "flavour": "plain", "mode": "partial"},
        # no reuse: a full setup in every step, the strategy that partial reuse
        # is compared with (and each series' first step)
        {"name": "rebuild_3d64", "kind": "poisson", "dim": 3, "N": 64, "precision": "fp64", "flavour": "sa", "mode": "rebuild"},
        # level-set transport (nonsymmetric): BiCGStab
        {"name": "levelset_3d64", "kind": "levelset", "dim": 3, "N": 64, "precision": "fp64"},
        # monolithic Navier-Stokes stand-in: 4 x 4 blocks, BiCGStab; about the
        # size of the paper's system (417,604 unknowns)
        {"name": "stokes_48", "kind": "stokes", "N": 48},
        # differentiable solve: forward and backward through the autograd function
        {"name": "grad_3d64", "kind": "grad", "dim": 3, "N": 64, "precision": "fp64"},
        # a simulation on the host: values and right-hand side come from, and the
        # solution goes to, pinned host buffers
        {"name": "host_3d128_mixed", "kind": "host", "dim": 3, "N": 128, "precision": "mixed"},
        # an unstructured matrix (rows of about 15 entries in a mesh-like
        # numbering, as from P1 elements)
        {"name": "mesh_41", "kind": "mesh", "N": 41, "precision": "fp64"},
    ]


def _between(rng, lo, hi):
    """A whole number, spread over its logarithm, odd or even alike."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["step2", "step3", "step3", "mixed", "mixed", "plain", "rebuild", "levelset", "stokes", "grad", "host",
                       "mesh"])
    prec = rng.choice(["fp64", "mixed"])
    if kind == "step2":
        return {"kind": "poisson", "dim": 2, "N": _between(rng, 24, 400), "precision": prec, "flavour": "sa", "mode": "partial"}
    if kind == "step3":
        return {"kind": "poisson", "dim": 3, "N": _between(rng, 14, 100), "precision": "fp64", "flavour": "sa", "mode": "partial"}
    if kind == "mixed":
        return {"kind": "poisson", "dim": 3, "N": _between(rng, 40, 180), "precision": "mixed", "flavour": "sa", "mode": "partial"}
    if kind == "plain":
        return {"kind": "poisson", "dim": 3, "N": _between(rng, 20, 75), "precision": prec, "flavour": "plain", "mode": "partial"}
    if kind == "rebuild":
        return {"kind": "poisson", "dim": 3, "N": _between(rng, 20, 120), "precision": prec, "flavour": "sa", "mode": "rebuild"}
    if kind == "levelset":
        return {"kind": "levelset", "dim": 3, "N": _between(rng, 20, 110), "precision": prec}
    if kind == "stokes":
        return {"kind": "stokes", "N": _between(rng, 16, 52)}
    if kind == "grad":
        return {"kind": "grad", "dim": 3, "N": _between(rng, 20, 80), "precision": prec}
    if kind == "host":
        return {"kind": "host", "dim": 3, "N": _between(rng, 32, 140), "precision": "mixed"}
    return {"kind": "mesh", "N": _between(rng, 16, 56), "precision": prec}


# ------------------------------------------------------------------ fields
def _dev():
    return torch.device("cuda", torch.cuda.current_device())


def _gen(seed):
    g = torch.Generator(device=_dev())
    g.manual_seed(int(seed) & 0x7FFFFFFF)
    return g


def _front(seed):
    """The step that the seed stands for, in the first fifth of the series."""
    return 1 + int(seed) * 7 % (STEPS // 5)


def _density(dim, N, k):
    """Density of step k per cell, shaped (z,) y, x: 1000 in the water column."""
    c = (torch.arange(N, dtype=torch.float64, device=_dev()) + 0.5) / N
    a = 0.25 + 0.5 * k / STEPS
    inx, inh = c < a, c < 0.125 / a
    if dim == 2:
        m = inh[:, None] & inx[None, :]
    else:
        m = (inh[:, None, None] & inx[None, None, :]).expand(N, N, N)
    return torch.where(m, 1000.0, 1.0).to(torch.float64).contiguous()


def _rhs(n, seed):
    return torch.rand(n, generator=_gen(seed * 2 + 1), dtype=torch.float64, device=_dev()) * 2.0 - 1.0


def _faces(dim, N, k):
    """Face velocities of a rotating, divergence-free flow without flow through
    the walls, Courant number 2, its strength that of step k."""
    c = (torch.arange(N, dtype=torch.float64, device=_dev()) + 0.5) / N
    e = torch.arange(N + 1, dtype=torch.float64, device=_dev()) / N
    s = 2.0 * (1.0 + 0.5 * math.sin(2.0 * math.pi * k / STEPS))
    pi = math.pi
    fx = -torch.sin(pi * e)[None, None, :] * torch.cos(pi * c)[:, None, None] * torch.ones_like(c)[None, :, None]
    fy = torch.zeros(N, N + 1, N, dtype=torch.float64, device=_dev())
    fz = torch.cos(pi * c)[None, None, :] * torch.sin(pi * e)[:, None, None] * torch.ones_like(c)[None, :, None]
    return (s * fx).contiguous(), fy, (s * fz).contiguous()


def _log_density(dim, N, seed):
    """theta = log rho of the first step, with noise N(0, 0.1^2) per cell."""
    th = _density(dim, N, 0).log().reshape(-1)
    return th + 0.1 * torch.randn(th.numel(), generator=_gen(seed * 2 + 2), dtype=torch.float64, device=_dev())


def _mesh(N, seed):
    """An unstructured symmetric pattern on N^3 nodes: every node is coupled to
    its face neighbours and to some of the other neighbours of a 3^3 box, and
    the nodes are numbered at random within windows of 256.  Returns CSR ptr,
    col, and per entry its edge's length factor and its two end nodes' cells
    (-1 factors mark the diagonal)."""
    n = N ** 3
    g = _gen(seed * 2 + 5)
    dev = _dev()
    idx = torch.arange(n, device=dev).reshape(N, N, N)
    ei, ej, ew = [], [], []
    for dz in (-1, 0, 1):
        for dy in (-1, 0, 1):
            for dx in (-1, 0, 1):
                if (dz, dy, dx) <= (0, 0, 0):
                    continue

                def cut(d):
                    return slice(0, N - d) if d >= 0 else slice(-d, N), slice(d, N) if d >= 0 else slice(0, N + d)

                (z0, z1), (y0, y1), (x0, x1) = cut(dz), cut(dy), cut(dx)
                a, b = idx[z0, y0, x0].reshape(-1), idx[z1, y1, x1].reshape(-1)
                keep = torch.rand(a.numel(), generator=g, device=dev) < (1.0 if abs(dz) + abs(dy) + abs(dx) == 1 else 0.4)
                w = 0.5 + 0.5 * torch.rand(a.numel(), generator=g, dtype=torch.float64, device=dev)
                ei.append(a[keep])
                ej.append(b[keep])
                ew.append(w[keep])
    ei, ej, ew = torch.cat(ei), torch.cat(ej), torch.cat(ew)
    key = torch.arange(n, device=dev) // 256 + torch.rand(n, generator=g, dtype=torch.float64, device=dev)
    order = torch.argsort(key)            # new number -> cell
    number = torch.empty_like(order)
    number[order] = torch.arange(n, device=dev)
    rows = torch.cat([number[ei], number[ej], torch.arange(n, device=dev)])
    cols = torch.cat([number[ej], number[ei], torch.arange(n, device=dev)])
    fac = torch.cat([ew, ew, torch.full((n,), -1.0, dtype=torch.float64, device=dev)])
    by = torch.argsort(rows * n + cols)
    rows, cols, fac = rows[by], cols[by], fac[by]
    ptr = torch.zeros(n + 1, dtype=torch.int64, device=dev)
    ptr[1:] = torch.cumsum(torch.bincount(rows, minlength=n), 0)
    return ptr.to(torch.int32), cols.to(torch.int32), rows, cols, fac, order


def _mesh_values(N, k, rows, cols, fac, order):
    """Values of step k on that pattern: minus the edge's factor times the
    harmonic coefficient, the diagonal so that rows sum to zero but for the top
    layer, where the pressure is held."""
    n = N ** 3
    rho = _density(3, N, k).reshape(-1)[order]
    off = fac > 0
    w = torch.where(off, fac * 2.0 / (rho[rows] + rho[cols]), torch.zeros_like(fac))
    dia = torch.segment_reduce(w, "sum", lengths=torch.bincount(rows, minlength=n))
    dia = dia + torch.where(order >= n - N * N, 2.0 / rho, torch.zeros_like(rho))
    return torch.where(off, -w, dia[rows]).contiguous()


# ------------------------------------------------------------------ states
def _params(case):
    kw = {"precision": B.PREC_MIXED if case.get("precision") == "mixed" else B.PREC_FP64}
    if case.get("flavour") == "plain":
        kw.update(smoothed=0, smoother=B.SMOOTHER_JACOBI)
    if case.get("mode") == "rebuild":
        kw.update(mode=B.MODE_FULL_REBUILD)
    if case["kind"] == "levelset":
        kw.update(solver=B.SOLVER_BICGSTAB)
    return kw


def prepare(case, seed):
    kind, N, k = case["kind"], case["N"], _front(seed)
    dim = case.get("dim", 3)
    n = N ** dim
    s = {"kind": kind, "dim": dim, "N": N}
    if kind == "grad":
        s["solver"] = AD.PoissonSolver(dim, N, tol=GRAD_TOL, **_params(case))
        s["theta"] = _log_density(dim, N, seed).requires_grad_(True)
        s["f"] = _rhs(n, seed).requires_grad_(True)
        s["target"] = torch.zeros(n, dtype=torch.float64, device=_dev())
        run(s)  # the first forward and backward pass of the optimisation
        return s
    if kind == "mesh":
        ptr, col, *mesh = _mesh(N, seed)
        s["amg"] = B.AMG(**_params(case))
        s["f"], s["u"] = _rhs(n, seed), torch.empty(n, dtype=torch.float64, device=_dev())
        s["amg"].step(_mesh_values(N, 0, *mesh), ptr, col)
        s["val"] = _mesh_values(N, k, *mesh)
        run(s)
        return s
    ptr, col = B.poisson_pattern(dim, N)
    s["ptr"] = ptr
    if kind == "stokes":
        s["amg"] = B.AMG(B.block_params())
        s["f"], s["u"] = _rhs(4 * n, seed), torch.empty(4 * n, dtype=torch.float64, device=_dev())
        first = _stokes_fields(N, 0)
        s["fields"] = _stokes_fields(N, k)
        s["val"] = B.stokes_values(N, *first, 0.1, ptr)
    elif kind == "levelset":
        s["amg"] = B.AMG(**_params(case))
        s["f"], s["u"] = _rhs(n, seed), torch.empty(n, dtype=torch.float64, device=_dev())
        s["faces"] = _faces(dim, N, k)
        s["val"] = B.levelset_values(dim, N, *_faces(dim, N, 0), ptr)
    else:
        s["amg"] = B.AMG(**_params(case))
        s["f"], s["u"] = _rhs(n, seed), torch.empty(n, dtype=torch.float64, device=_dev())
        s["rho"] = _density(dim, N, k)
        s["val"] = B.poisson_values(dim, N, _density(dim, N, 0), ptr)
    s["amg"].step(s["val"], ptr, col)
    if kind == "host":
        val = B.poisson_values(dim, N, s["rho"], ptr)
        s["h_val"] = torch.empty(val.numel(), dtype=torch.float64, pin_memory=True).copy_(val).numpy()
        s["h_f"] = torch.empty(n, dtype=torch.float64, pin_memory=True).copy_(s["f"]).numpy()
        s["h_u"] = torch.zeros(n, dtype=torch.float64, pin_memory=True).numpy()
    run(s)  # the series' second step
    return s


def _stokes_fields(N, k):
    rho = _density(3, N, k)
    mu = torch.where(rho == 1000.0, 1.0, 0.018).to(torch.float64).contiguous()
    return (rho, mu, *_faces(3, N, k))


def run(s):
    kind = s["kind"]
    if kind == "grad":
        u = AD.solve(s["theta"], s["f"], s["solver"])
        loss = 0.5 * ((u - s["target"]) ** 2).sum()
        g_theta, g_f = torch.autograd.grad(loss, (s["theta"], s["f"]))
        return {"u": u.detach(), "theta": g_theta, "f": g_f}
    if kind == "host":
        s["amg"].step_solve_host(s["h_val"], s["h_f"], s["h_u"], TOL)
        return {"u": s["h_u"]}
    if kind == "poisson":
        B.poisson_values(s["dim"], s["N"], s["rho"], s["ptr"], out=s["val"])
    elif kind == "levelset":
        B.levelset_values(s["dim"], s["N"], *s["faces"], s["ptr"], out=s["val"])
    elif kind == "stokes":
        B.stokes_values(s["N"], *s["fields"], 0.1, s["ptr"], out=s["val"])
    s["amg"].step(s["val"])
    u, _ = s["amg"].solve(s["f"], TOL, u=s["u"])
    return {"u": u}


def work(case):
    """The step's inputs read once and its solution written once: the fields
    (or values) that the matrix comes from, the pattern, the right-hand side;
    the operations of one product with the matrix."""
    N, kind = case["N"], case["kind"]
    dim = case.get("dim", 3)
    n = N ** dim
    nnz = n + 2 * dim * (N - 1) * N ** (dim - 1)
    if kind == "mesh":
        nnz = int(n * 15.0)
        return {"bytes": 12 * nnz + 4 * n + 16 * n, "flops": 2 * nnz}
    if kind == "stokes":
        return {"bytes": 4 * nnz + 4 * n + 8 * 5 * n + 64 * n, "flops": 32 * nnz}
    if kind == "grad":
        return {"bytes": 4 * nnz + 4 * n + 8 * 6 * n, "flops": 4 * nnz}
    if kind == "host":
        return {"bytes": 12 * nnz + 4 * n + 16 * n, "flops": 2 * nnz}
    fields = 3 if kind == "levelset" else 1
    return {"bytes": 4 * nnz + 4 * n + 8 * fields * n + 16 * n, "flops": 2 * nnz}


# ------------------------------------------------------------------ in 64 bits, plain torch
def _shift_sum(parts, x, dim):
    """Sum over the faces: parts holds, per axis, the (low, high) coefficients
    of the neighbours along it (zero where there is none)."""
    y = torch.zeros_like(x)
    for ax, (lo, hi) in enumerate(parts):
        m = x.shape[ax]
        y.narrow(ax, 1, m - 1).add_(lo.narrow(ax, 1, m - 1) * x.narrow(ax, 0, m - 1))
        y.narrow(ax, 0, m - 1).add_(hi.narrow(ax, 0, m - 1) * x.narrow(ax, 1, m - 1))
    return y


def _pcg(apply, dia, f, tol=1e-14, most=6000):
    u = torch.zeros_like(f)
    r, z = f.clone(), f / dia
    p, rz, nf = z.clone(), (f * (f / dia)).sum(), f.norm()
    best, best_u = float("inf"), u.clone()
    for it in range(most):
        q = apply(p)
        alpha = rz / (p * q).sum()
        u += alpha * p
        r -= alpha * q
        if it % 25 == 24:
            res = float(r.norm() / nf)
            if res < best:
                best, best_u = res, u.clone()
            if res < tol or not math.isfinite(res):
                break
        z = r / dia
        new = (r * z).sum()
        p = z + (new / rz) * p
        rz = new
    return best_u


def _poisson_parts(rho):
    """(per-axis neighbour coefficients, diagonal) of -div((1/rho) grad p) with
    harmonic face coefficients, p = 0 beyond the top."""
    dim = rho.dim()
    parts, dia = [], torch.zeros_like(rho)
    for ax in range(dim):
        m = rho.shape[ax]
        k = 2.0 / (rho.narrow(ax, 0, m - 1) + rho.narrow(ax, 1, m - 1))
        lo, hi = torch.zeros_like(rho), torch.zeros_like(rho)
        lo.narrow(ax, 1, m - 1).copy_(-k)
        hi.narrow(ax, 0, m - 1).copy_(-k)
        dia -= lo + hi
        parts.append((lo, hi))
    dia[-1] += 2.0 / rho[-1]
    return parts, dia


def _poisson_solve(rho, f):
    parts, dia = _poisson_parts(rho)
    dim = rho.dim()
    return _pcg(lambda x: dia * x + _shift_sum(parts, x, dim), dia, f.reshape(rho.shape)).reshape(-1)


def _log_gradient(rho, u, lam):
    """dL/dlog(rho) from A lam = dL/du: the chain through the face coefficients
    k = 2 / (rho_i + rho_j) and the top's 2 / rho_i."""
    u, lam = u.reshape(rho.shape), lam.reshape(rho.shape)
    g = torch.zeros_like(rho)
    for ax in range(rho.dim()):
        m = rho.shape[ax]
        a, b = rho.narrow(ax, 0, m - 1), rho.narrow(ax, 1, m - 1)
        du = u.narrow(ax, 0, m - 1) - u.narrow(ax, 1, m - 1)
        dl = lam.narrow(ax, 0, m - 1) - lam.narrow(ax, 1, m - 1)
        dk = -2.0 / (a + b) ** 2 * (-dl * du)
        g.narrow(ax, 0, m - 1).add_(dk * a)
        g.narrow(ax, 1, m - 1).add_(dk * b)
    g[-1] += (-lam[-1] * u[-1]) * (-2.0 / rho[-1])
    return g.reshape(-1)


def _bicgstab(apply, prec, f, tol=1e-14, most=4000):
    x = torch.zeros_like(f)
    r, rh = f.clone(), f.clone()
    rho = alpha = omega = torch.ones((), dtype=f.dtype, device=f.device)
    v, p, nf = torch.zeros_like(f), torch.zeros_like(f), f.norm()
    best, best_x = float("inf"), x.clone()
    for it in range(most):
        new = (rh * r).sum()
        p = r + (new / rho) * (alpha / omega) * (p - omega * v)
        rho = new
        ph = prec(p)
        v = apply(ph)
        alpha = rho / (rh * v).sum()
        s = r - alpha * v
        sh = prec(s)
        t = apply(sh)
        omega = (t * s).sum() / (t * t).sum()
        x = x + alpha * ph + omega * sh
        r = s - omega * t
        if it % 10 == 9:
            res = float((f - apply(x)).norm() / nf)
            if res < best:
                best, best_x = res, x.clone()
            if res < tol or not math.isfinite(res) or res > 1e6 * best:
                break
    return best_x


def _levelset_solve(N, faces, f):
    """The upwind system: off-diagonal min(w, 0) - 0.1 per face with w the
    outward flux, diagonal 1 + sum of max(w, 0) + 0.1; Jacobi iterations."""
    fx, fy, fz = faces
    parts, dia = [], torch.ones(N, N, N, dtype=torch.float64, device=f.device)
    for ax, v in enumerate((fz, fy, fx)):
        lo_w, hi_w = -v.narrow(ax, 0, N), v.narrow(ax, 1, N)
        lo, hi = torch.clamp(lo_w, max=0.0) - 0.1, torch.clamp(hi_w, max=0.0) - 0.1
        inner = torch.ones_like(dia)
        inner.narrow(ax, 0, 1).zero_()
        dia += inner * (torch.clamp(lo_w, min=0.0) + 0.1)
        lo = lo * inner
        inner = torch.ones_like(dia)
        inner.narrow(ax, N - 1, 1).zero_()
        dia += inner * (torch.clamp(hi_w, min=0.0) + 0.1)
        hi = hi * inner
        parts.append((lo, hi))
    return _bicgstab(lambda x: dia * x + _shift_sum(parts, x, 3), lambda x: x / dia, f.reshape(N, N, N)).reshape(-1)


def _stokes_solve(N, fields, f, mass=0.1):
    """The 4 x 4 block system, matrix-free (velocities u, v, w along x, y, z and
    the pressure), solved by BiCGStab with the blocks' inverses."""
    rho, mu, fx, fy, fz = fields
    kap = mass * rho + 6.0 * mu
    dia_v, dia_p = mass * rho.clone(), torch.zeros_like(rho)
    wall = [torch.zeros_like(rho) for _ in range(3)]      # (u_d, p) of the diagonal block, d = x, y, z
    vel, pres, cpl = [], [], []
    for ax, v in enumerate((fz, fy, fx)):
        two_v, two_p, two_c = [], [], []
        for side, (at, to) in ((-1, (1, 0)), (1, (0, 1))):
            phi = side * v.narrow(ax, 0 if side < 0 else 1, N)
            m_c, m_j = mu.narrow(ax, at, N - 1), mu.narrow(ax, to, N - 1)
            k_c, k_j = kap.narrow(ax, at, N - 1), kap.narrow(ax, to, N - 1)
            muf = 2.0 * m_c * m_j / (m_c + m_j)
            beta = 2.0 / (1.0 / k_c + 1.0 / k_j)
            ph = phi.narrow(ax, at, N - 1)
            full = [torch.zeros_like(rho) for _ in range(3)]
            full[0].narrow(ax, at, N - 1).copy_(torch.clamp(ph, max=0.0) - muf)
            full[1].narrow(ax, at, N - 1).copy_(-beta)
            full[2].narrow(ax, at, N - 1).copy_(0.5 * side * beta)
            dia_v.narrow(ax, at, N - 1).add_(muf + torch.clamp(ph, min=0.0))
            dia_p.narrow(ax, at, N - 1).add_(beta)
            edge = 0 if side < 0 else N - 1
            dia_v.narrow(ax, edge, 1).add_(2.0 * mu.narrow(ax, edge, 1))
            wall[2 - ax].narrow(ax, edge, 1).add_(0.5 * side * kap.narrow(ax, edge, 1))
            two_v.append(full[0])
            two_p.append(full[1])
            two_c.append(full[2])
        vel.append(tuple(two_v))
        pres.append(tuple(two_p))
        cpl.append(tuple(two_c))
    dia_p[-1] += 2.0 * kap[-1]

    def apply(x):
        y = torch.empty_like(x)
        p = x[3]
        y[3] = dia_p * p + _shift_sum(pres, p, 3)
        zero = (torch.zeros_like(rho), torch.zeros_like(rho))
        for d in range(3):
            only = [cpl[ax] if 2 - ax == d else zero for ax in range(3)]
            y[d] = dia_v * x[d] + _shift_sum(vel, x[d], 3) + wall[d] * p + _shift_sum(only, p, 3)
            y[3] += _shift_sum(only, x[d], 3) - wall[d] * x[d]
        return y

    D = torch.zeros(N, N, N, 4, 4, dtype=torch.float64, device=f.device)
    for d in range(3):
        D[..., d, d] = dia_v
        D[..., d, 3] = wall[d]
        D[..., 3, d] = -wall[d]
    D[..., 3, 3] = dia_p
    inv = torch.linalg.inv(D)
    x = _bicgstab(apply, lambda t: torch.einsum("zyxij,jzyx->izyx", inv, t),
                  f.reshape(N, N, N, 4).permute(3, 0, 1, 2).contiguous())
    return x.permute(1, 2, 3, 0).reshape(-1)


def exact(case, seed):
    kind, N, k = case["kind"], case["N"], _front(seed)
    dim = case.get("dim", 3)
    n = N ** dim
    if kind == "grad":
        rho = _log_density(dim, N, seed).exp().reshape((N,) * dim)
        u = _poisson_solve(rho, _rhs(n, seed))
        lam = _poisson_solve(rho, u)
        return {"u": u, "theta": _log_gradient(rho, u, lam), "f": lam}
    if kind == "mesh":
        ptr, col, *mesh = _mesh(N, seed)
        val = _mesh_values(N, k, *mesh)
        A = torch.sparse_csr_tensor(ptr, col, val, size=(n, n))
        rows, cols = mesh[0], mesh[1]
        return {"u": _pcg(lambda x: torch.mv(A, x), val[rows == cols], _rhs(n, seed))}
    if kind == "levelset":
        return {"u": _levelset_solve(N, _faces(dim, N, k), _rhs(n, seed))}
    if kind == "stokes":
        return {"u": _stokes_solve(N, _stokes_fields(N, k), _rhs(4 * n, seed))}
    return {"u": _poisson_solve(_density(dim, N, k), _rhs(n, seed))}
