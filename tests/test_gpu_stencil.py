"""The finest level by diagonals (patterns of at most eight column offsets that
the rows fill to three quarters) against the oracle, at the edges of its range:
one to eight offsets, ragged row counts, rows with absent entries, and the
first patterns on the other side of the rule, which stay in CSR."""
import numpy as np
import pytest
import scipy.sparse as sp

import oracle as O
from paper_2108_02054_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2108_02054_gb300 import amg as B

SYM = {3: (-1, 1), 5: (-7, -1, 1, 7), 7: (-40, -6, -1, 1, 6, 40), 9: (-40, -6, -2, -1, 1, 2, 6, 40)}


def stencil_matrix(n, offsets, keep, seed):
    """Diagonally dominant symmetric values on row + offsets, a share `keep` of
    the entries present."""
    rng = np.random.default_rng(seed)
    M = sp.csr_matrix((n, n))
    for d in offsets:
        if d <= 0 or d >= n:
            continue
        i = np.arange(n - d)
        i = i[rng.random(i.size) < keep]
        w = -rng.uniform(0.1, 1.0, i.size)
        M = M + sp.csr_matrix((w, (i, i + d)), (n, n))
    M = (M + M.T).tocsr()
    M = M + sp.diags(-np.asarray(M.sum(axis=1)).ravel() + rng.uniform(0.01, 0.5, n))
    M = M.tocsr()
    M.sort_indices()
    return M.indptr.astype(np.int32), M.indices.astype(np.int32), M.data.astype(np.float64)


def cuda(*a):
    return tuple(torch.tensor(x, device="cuda") for x in a)


@pytest.mark.parametrize("noff,n,keep", [(3, 33, 1.0), (3, 1001, 0.95), (5, 1024, 1.0), (5, 5003, 0.9), (7, 997, 1.0),
                                         (7, 20011, 0.9), (7, 4000, 0.6), (9, 3001, 1.0)])
def test_stencil_forms_against_oracle(noff, n, keep):
    ptr, col, val = stencil_matrix(n, SYM[noff], keep, seed=noff * 1000 + n)
    G = B.AMG(coarse_enough=20)
    G.full_setup(*cuda(ptr, col, val))
    assert G.pattern_info() == (1, noff)
    H = O.Hierarchy(ptr, col, val, O.Params(coarse_enough=20))
    new = I.revalue_symmetric(ptr, col, val, seed=5)
    G.partial_rebuild(cuda(new)[0])
    H.rebuild(new)
    assert G.nlevels == H.nlevels
    for l in range(H.nlevels):  # the exported values are the new ones, bit for bit
        assert np.array_equal(G.export_level(l)["A"][2], H.level(l).A.val)
    r = np.random.default_rng(3).normal(size=n)
    z, zo = G.vcycle(cuda(r)[0]).cpu().numpy(), H.vcycle(r)
    # FP64 sums of the same terms in another order at most
    assert np.linalg.norm(z - zo) <= 1e-11 * np.linalg.norm(zo)
    u, info = G.solve(cuda(r)[0], 1e-8)
    _, it, _, st = H.pcg(r, 1e-8)
    assert info.status == 0 and st == 0 and abs(info.iters - it) <= 1
    A = sp.csr_matrix((new, col, ptr))
    assert np.linalg.norm(r - A @ u.cpu().numpy()) <= 1.001e-8 * np.linalg.norm(r)


@pytest.mark.parametrize("n", [1001, 60000, 100000, 160001])
def test_stencil_mixed_orders(n):
    """FP32 rows in the order of 8, 4, 2 and 1 lanes (by size): the V-cycle
    against the FP64 oracle.  FP32 rounding of a cycle's few products is below
    1e-5 of z."""
    ptr, col, val = stencil_matrix(n, SYM[7], 0.95, seed=n)
    G = B.AMG(precision=B.PREC_MIXED)
    G.full_setup(*cuda(ptr, col, val))
    H = O.Hierarchy(ptr, col, val)
    r = np.random.default_rng(3).normal(size=n)
    z, zo = G.vcycle(cuda(r)[0]).cpu().numpy(), H.vcycle(r)
    assert np.linalg.norm(z - zo) <= 1e-5 * np.linalg.norm(zo)
    u, info = G.solve(cuda(r)[0], 1e-8)
    assert info.status == 0 and info.rel_resid <= 1e-8


@pytest.mark.parametrize("noff", [7, 8])
def test_stencil_bicgstab_and_full_reuse(noff):
    """A nonsymmetric stencil (eight offsets: one diagonal without its
    transpose) through BiCGStab in full-reuse mode, where the system matrix is
    apart from the hierarchy's."""
    n = 3001
    ptr, col, val = stencil_matrix(n, SYM[7], 1.0, seed=8)
    A = sp.csr_matrix((val, col, ptr)).tolil()
    if noff == 8:
        for i in range(0, n - 90):
            A[i, i + 90] = -0.01
    A = A.tocsr()
    A.sort_indices()
    ptr, col, val = A.indptr.astype(np.int32), A.indices.astype(np.int32), A.data
    G = B.AMG(solver=B.SOLVER_BICGSTAB, mode=B.MODE_FULL_REUSE)
    f = np.random.default_rng(4).normal(size=n)
    G.step(cuda(val)[0], *cuda(ptr, col))
    assert G.pattern_info() == (1, noff)
    for scale in (1.0, 1.25):
        G.step(cuda(val * scale)[0])
        u, info = G.solve(cuda(f)[0], 1e-9)
        assert info.status == 0
        assert np.linalg.norm(f - scale * (A @ u.cpu().numpy())) <= 1.01e-9 * np.linalg.norm(f)


@pytest.mark.parametrize("maxiter,precision,nlev1", [(1, 0, False), (2, 0, False), (7, 0, False), (1, 1, False),
                                                     (6, 1, False), (1, 0, True), (1, 1, True)])
def test_iterate_when_maxiter_ends_it(maxiter, precision, nlev1):
    """u += alpha p is part of the p update except where the iteration ends:
    the iterate left by maxiter against the oracle's, FP64 (1e-10) and with an
    FP32 cycle (its rounding, 1e-4), with and without a coarse level."""
    n = 1000
    ptr, col, val = stencil_matrix(n, SYM[5], 1.0, seed=maxiter)
    kw = dict(coarse_enough=n if nlev1 else 50)
    f = np.random.default_rng(6).normal(size=n)
    G = B.AMG(precision=precision, maxiter=maxiter, **kw)
    G.full_setup(*cuda(ptr, col, val))
    u, info = G.solve(cuda(f)[0], 1e-30)
    H = O.Hierarchy(ptr, col, val, O.Params(**kw))
    uo, it, rr, st = H.pcg(f, 1e-30, maxiter=maxiter)
    assert info.iters == it and info.status != 0 and st != 0
    assert np.linalg.norm(u.cpu().numpy() - uo) <= (1e-10 if precision == 0 else 1e-4) * np.linalg.norm(uo)
