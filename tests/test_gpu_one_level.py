"""Hierarchies of one level (the finest is the coarsest: small systems,
max_levels = 1, coarsening that stalls) after new values: the factors, the
V-cycle (then the exact solve) and the iteration count against the oracle,
through every entry point that refreshes the values."""
import numpy as np
import pytest

import oracle as O
from paper_2108_02054_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2108_02054_gb300 import amg as B
    from paper_2108_02054_gb300 import autograd as AD

EPS = np.finfo(np.float64).eps
STEPS = 4


def cuda(a):
    return torch.tensor(a, device="cuda")


def problem(kind):
    """ptr, col, values of two steps and the options of the one-level hierarchy."""
    if kind in ("2d16", "2d5", "3d6", "max_levels"):
        dim, N = {"2d16": (2, 16), "2d5": (2, 5), "3d6": (3, 6), "max_levels": (2, 24)}[kind]
        ptr, col, v0 = O.poisson_assemble(dim, N, I.density(dim, N, 0, STEPS))
        v1 = O.poisson_assemble(dim, N, I.density(dim, N, STEPS - 1, STEPS))[2]
        return ptr, col, v0, v1, {"max_levels": 1} if kind == "max_levels" else {}
    # no strong couplings at all: the first level cannot be coarsened
    n = 300
    i = np.arange(n)
    ptr = np.concatenate([[0], np.cumsum(np.where((i == 0) | (i == n - 1), 2, 3))]).astype(np.int32)
    col = np.concatenate([[j for j in (k - 1, k, k + 1) if 0 <= j < n] for k in i]).astype(np.int32)
    row = np.repeat(i, np.diff(ptr))
    rng = np.random.default_rng(2)
    d0, d1 = rng.uniform(1.0, 2.0, n), rng.uniform(1.0, 2.0, n)
    return ptr, col, np.where(row == col, d0[row], -0.01), np.where(row == col, d1[row], -0.01), {}


def pcg_iterations(A, P, f, tol):
    """CG preconditioned by a dense solve with P: iterations to the tolerance."""
    inv = np.linalg.inv(P)
    u, r = np.zeros_like(f), f.copy()
    p = z = inv @ r
    for it in range(1, 100):
        q = A @ p
        rz = r @ z
        alpha = rz / (p @ q)
        u, r = u + alpha * p, r - alpha * q
        if np.linalg.norm(r) <= tol * np.linalg.norm(f):
            return it
        z = inv @ r
        p = z + (r @ z) / rz * p
    return it


def dense(ptr, col, val):
    n = ptr.size - 1
    M = np.zeros((n, n))
    M[np.repeat(np.arange(n), np.diff(ptr)), col] = val
    return M


KINDS = ["2d16", "2d5", "3d6", "max_levels", "stalled"]


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("solver", [0, 1])
@pytest.mark.parametrize("entry", ["partial_rebuild", "step", "host"])
@pytest.mark.parametrize("kind", KINDS)
def test_new_values_reach_the_factors(kind, entry, solver, precision):
    ptr, col, v0, v1, kw = problem(kind)
    n = ptr.size - 1
    G = B.AMG(solver=solver, precision=precision, **kw)
    G.full_setup(cuda(ptr), cuda(col), cuda(v0))
    assert G.nlevels == 1
    f = I.rhs(n)
    for v in (v1, v0, v1):
        if entry == "host":
            u = np.empty(n)
            info = G.step_solve_host(v, f, u, 1e-8)
            assert info.rebuilt == 0
        else:
            if entry == "step":
                assert G.step(cuda(v)).rebuilt == 0
            else:
                G.partial_rebuild(cuda(v))
            u, info = G.solve(cuda(f), 1e-8)
            u = u.cpu().numpy()
        # the factorised matrix: the new values, in FP32 under mixed precision
        vf = v.astype(np.float32).astype(np.float64) if precision else v
        assert np.array_equal(G.export_level(0)["A"][2], vf)
        A, M = dense(ptr, col, v), dense(ptr, col, vf)
        olu, opiv, ost = O.dense_lu(M)
        lu, piv = G.coarse_lu()
        assert ost == O.OK and np.array_equal(piv, opiv)
        assert np.allclose(lu, olu, rtol=1e-12, atol=1e-14 * np.abs(olu).max())
        # the cycle is the explicit inverse times r: n eps cond
        z, ref = G.vcycle(cuda(f)).cpu().numpy(), np.linalg.solve(M, f)
        assert np.linalg.norm(z - ref) <= 10 * n * EPS * np.linalg.cond(M) * np.linalg.norm(ref)
        # (a BiCGStab iteration applies the cycle twice)
        it = pcg_iterations(A, M, f, 1e-8)
        assert info.status == 0 and info.iters <= it + 1, (info.iters, it)
        assert np.linalg.norm(f - A @ u) <= 1.001e-8 * np.linalg.norm(f)


@pytest.mark.parametrize("entry", ["partial_rebuild", "step", "host"])
def test_a_matrix_that_became_singular_is_refused(entry):
    ptr, col, v0, v1, kw = problem("2d16")
    n = ptr.size - 1
    G = B.AMG(**kw)
    G.full_setup(cuda(ptr), cuda(col), cuda(v0))
    row = np.repeat(np.arange(n), np.diff(ptr))
    bad = np.where((row == 40) | (col == 40), 0.0, v1)
    with pytest.raises(B.AmgError) as e:
        if entry == "host":
            G.step_solve_host(bad, I.rhs(n), np.empty(n))
        elif entry == "step":
            G.step(cuda(bad))
        else:
            G.partial_rebuild(cuda(bad))
    assert e.value.status == B.AMG_ERR_SINGULAR


@pytest.mark.parametrize("dim,N", [(2, 16), (3, 6)])
def test_differentiable_solve_with_changing_theta(dim, N):
    S = AD.PoissonSolver(dim, N)
    n = N ** dim
    f = torch.tensor(I.rhs(n), device="cuda")
    for k in (0, 3, 1):
        theta = torch.tensor(np.log(I.density(dim, N, k, STEPS)).ravel(), device="cuda", requires_grad=True)
        u = AD.solve(theta, f, S)
        u.sum().backward()
        A = dense(*O.poisson_assemble(dim, N, np.exp(theta.detach().cpu().numpy())))
        assert S.amg.nlevels == 1
        assert S.last_info.iters <= pcg_iterations(A, A, f.cpu().numpy(), S.tol) + 1
        assert S.adjoint_info.iters <= pcg_iterations(A, A, np.ones(n), S.tol) + 1
        r = f.cpu().numpy() - A @ u.detach().cpu().numpy()
        assert np.linalg.norm(r) <= 1.001e-10 * np.linalg.norm(f.cpu().numpy())
