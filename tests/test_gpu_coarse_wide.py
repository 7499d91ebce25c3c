"""The coarsest LU between 128 and 256 rows (eight compute warps, message rows
in a ring that later steps reuse) and between 449 and 1,024 (panels of 16
columns), and their inverses, against the oracle."""
import numpy as np
import pytest

import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2108_02054_gb300 import amg as B


def dense(M):
    n = M.shape[0]
    return (torch.arange(0, n * n + 1, n, dtype=torch.int32, device="cuda"),
            torch.arange(n, dtype=torch.int32, device="cuda").repeat(n), torch.tensor(M.ravel(), device="cuda"))


@pytest.mark.parametrize("n", [129, 153, 159, 192, 224, 255, 256, 257, 449, 463, 464, 481, 511, 1009, 1023, 1024, 1025])
def test_factors_and_inverse(n):
    """Tied small-integer pivots: factors and pivots bit for bit, twice on one
    context (nothing is left behind), and the V-cycle (the inverse times r)
    against a dense solve to n eps cond."""
    rng = np.random.default_rng(n)
    M = rng.integers(-3, 4, (n, n)).astype(np.float64) + np.eye(n)
    olu, opiv, ost = O.dense_lu(M)
    assert ost == O.OK
    G = B.AMG(coarse_enough=n)
    for _ in range(2):
        G.full_setup(*dense(M))
        lu, piv = G.coarse_lu()
        assert np.array_equal(piv, opiv) and np.array_equal(lu, olu)
    r = rng.normal(size=n)
    z = G.vcycle(torch.tensor(r, device="cuda")).cpu().numpy()
    ref = np.linalg.solve(M, r)
    assert np.linalg.norm(z - ref) <= 10 * n * 2.3e-16 * np.linalg.cond(M) * np.linalg.norm(ref)


@pytest.mark.parametrize("n,j", [(255, j) for j in (0, 39, 40, 41, 127, 128, 200, 253, 254)]
                         + [(467, j) for j in (0, 1, 15, 16, 463, 464, 466)])
def test_zero_column(n, j):
    rng = np.random.default_rng(700 + j)
    M = rng.integers(-3, 4, (n, n)).astype(np.float64) + np.eye(n) * 20.0
    Z = M.copy()
    Z[:, j] = 0.0
    G = B.AMG(coarse_enough=n)
    with pytest.raises(B.AmgError) as e:
        G.full_setup(*dense(Z))
    assert e.value.status == B.AMG_ERR_SINGULAR
    olu, opiv, _ = O.dense_lu(M)
    G.full_setup(*dense(M))
    lu, piv = G.coarse_lu()
    assert np.array_equal(piv, opiv) and np.array_equal(lu, olu)
