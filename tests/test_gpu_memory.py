"""Device memory that a hierarchy holds after a setup, a step and a solve, at
128^3: no more than with the finest matrix held once in CSR and the setup's
scratch kept (a system that once fitted the device still fits)."""
import pytest

from paper_2108_02054_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2108_02054_gb300 import amg as B

N = 128
# (precision, mode, smoothed): MB measured with that layout
LIMITS = {(0, 0, 1): 4578, (1, 0, 1): 4194, (0, 1, 1): 1506, (1, 1, 1): 1666, (0, 2, 1): 1602, (1, 2, 1): 1794,
          (0, 0, 0): 1538, (1, 0, 0): 1506}


def held(precision, mode, smoothed):
    """MB, by the device's free memory before and after."""
    kw = dict(precision=precision, mode=mode, maxiter=200)
    if not smoothed:
        kw.update(smoothed=0, smoother=B.SMOOTHER_JACOBI)
    ptr, col = B.poisson_pattern(3, N)
    val = B.poisson_values(3, N, torch.tensor(I.density(3, N, 3, 10), device="cuda"), ptr)
    f = torch.ones(N ** 3, dtype=torch.float64, device="cuda")
    u = torch.empty_like(f)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    G = B.AMG(**kw)
    G.step(val, ptr, col)
    G.step(val)
    assert G.solve(f, 1e-6, u=u)[1].status == 0
    torch.cuda.synchronize()
    used = free - torch.cuda.mem_get_info()[0]
    assert G.pattern_info() == (1, 7)
    G.close()
    return used / 2 ** 20


@pytest.mark.parametrize("case", sorted(LIMITS))
def test_device_memory_of_a_hierarchy(case):
    held(*case)  # (first use: the runtime's own memory)
    assert held(*case) <= LIMITS[case]


def test_full_reuse_matrix_across_forms_of_one_size():
    """One context, patterns of the same rows and entries held by diagonals and
    in CSR in turn: the full-reuse system matrix is made again where its form
    needs more, and each solve is with the last step's values."""
    n = 600
    i = torch.arange(n - 1, device="cuda")
    G = B.AMG(mode=B.MODE_FULL_REUSE, coarse_enough=50)
    f = torch.linspace(-1.0, 1.0, n, dtype=torch.float64, device="cuda")
    for diagonals in (False, True, False, True, True):
        j = i + 1 if diagonals else torch.where(i + 1 + i % 7 < n, i + 1 + i % 7, i + 1)
        A = torch.eye(n, dtype=torch.float64, device="cuda") * 0.1
        for a, b in ((i, j), (j, i)):
            A.index_put_((a, b), torch.tensor(-1.0, dtype=torch.float64, device="cuda"))
            A.diagonal().index_add_(0, a, torch.ones(n - 1, dtype=torch.float64, device="cuda"))
        S = A.to_sparse_csr()
        ptr, col, val = S.crow_indices().int(), S.col_indices().int(), S.values().contiguous()
        assert val.numel() == 3 * n - 2
        G.full_setup(ptr, col, val)
        assert G.pattern_info() == (1, 3 if diagonals else 15)
        for scale in (1.0, 1.25):
            G.step(val * scale)
            u, info = G.solve(f, 1e-9)
            assert info.status == 0
            assert torch.linalg.norm(f - scale * (A @ u)) <= 1.01e-9 * torch.linalg.norm(f)
