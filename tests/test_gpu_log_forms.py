"""The log-density assembly and gradient on both sides of the rule that chooses
between the marching kernels and one thread per cell: values against the oracle,
and no size where the choice costs."""
import statistics

import numpy as np
import pytest

import oracle as O
from paper_2108_02054_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2108_02054_gb300 import amg as B


@pytest.mark.parametrize("top", [True, False])
@pytest.mark.parametrize("dim,N", [(2, 1), (2, 37), (2, 383), (2, 384), (2, 601), (3, 1), (3, 16), (3, 59), (3, 60), (3, 67)])
def test_both_forms_against_the_oracle(dim, N, top):
    n = N ** dim
    theta = I.noisy_log_density(dim, N, seed=4)
    ptr, _ = B.poisson_pattern(dim, N)
    th = torch.tensor(theta, device="cuda")
    v = B.poisson_values_log(dim, N, th, ptr, top).cpu().numpy()
    ref = O.poisson_assemble(dim, N, np.exp(theta), top)[2]
    # a density's exponential to an ulp or two, then a sum and a division a face
    assert np.allclose(v, ref, rtol=4e-16 * 8, atol=0)
    rng = np.random.default_rng(6)
    u, lam = rng.normal(size=n), rng.normal(size=n)
    g = B.poisson_grad_log(dim, N, th, torch.tensor(u, device="cuda"), torch.tensor(lam, device="cuda"), top)
    g_ref = O.poisson_grad_theta(dim, N, np.exp(theta), u, lam, top)
    assert np.allclose(g.cpu().numpy(), g_ref, rtol=1e-13, atol=1e-13 * np.abs(g_ref).max())


def device_us(call):
    """Device time of one call: twenty in a graph, the median of nine replays."""
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        call(s)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        for _ in range(20):
            call(s)
    times = []
    for _ in range(9):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        g.replay()
        b.record()
        b.synchronize()
        times.append(a.elapsed_time(b) * 50.0)
    return statistics.median(times)


@pytest.mark.parametrize("dim,N", [(2, 1024), (2, 1900), (3, 16), (3, 32), (3, 48)])
def test_time_beside_the_density_form(dim, N):
    """The faster form takes at most 3.1 times the assembly from densities at
    these sizes, the other one 4.6 to 8.8 times."""
    n = N ** dim
    ptr, _ = B.poisson_pattern(dim, N)
    th = torch.randn(n, dtype=torch.float64, device="cuda")
    rho = th.exp()
    out = torch.empty(B.poisson_nnz(dim, N), dtype=torch.float64, device="cuda")
    log = device_us(lambda s: B.poisson_values_log(dim, N, th, ptr, out=out, stream=s))
    lin = device_us(lambda s: B.poisson_values(dim, N, rho, ptr, out=out, stream=s))
    assert log <= 4.0 * lin, (log, lin)
