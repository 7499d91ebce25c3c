"""The setup's row kernels with a warp per row (more than eight entries a row
on average) against the oracle, where their pieces end: rows around 128, 256
and 512 entries (the sorting networks, the staged rows of P), aggregates of all
sizes, rows of one entry, and averages on both sides of the rule."""
import numpy as np
import pytest

import oracle as O
from paper_2108_02054_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2108_02054_gb300 import amg as B


def check(ptr, col, val, **kw):
    G = B.AMG(coarse_enough=12, **kw)
    G.full_setup(*(torch.tensor(a, device="cuda") for a in (ptr, col, val)))
    H = O.Hierarchy(ptr, col, val, O.Params(coarse_enough=12, **kw))
    assert G.nlevels == H.nlevels
    for l in range(H.nlevels):
        g, o = G.export_level(l), H.level(l)
        assert np.array_equal(g["agg"], o.agg) and np.array_equal(g["strong"], o.strong)
        assert np.array_equal(g["A"][1], o.A.col) and np.array_equal(g["A"][2], o.A.val)
        if l < H.nlevels - 1:
            for name, ref in (("P", o.P), ("R", o.R)):
                assert all(np.array_equal(x, y) for x, y in zip(g[name], (ref.ptr, ref.col, ref.val)))
    return G, H


@pytest.mark.parametrize("arm", [100, 130, 255, 258, 511, 514, 700])
def test_long_rows(arm):
    """One row and column of `arm` couplings: with weak couplings P's rows and
    R's stay short, with strong ones they span the arm."""
    n = 900
    for theta in (0.08, 0.0):
        ptr, col, val = I.random_arrow_spd(n, 0.012, arm, seed=arm)
        assert np.diff(ptr).max() >= arm
        check(ptr, col, val, theta=theta)


@pytest.mark.parametrize("density", [0.004, 0.007, 0.0085, 0.012, 0.1])
def test_both_sides_of_the_rule(density):
    n = 1000
    ptr, col, val = I.random_spd_like(n, density, seed=int(1e4 * density))
    G, H = check(ptr, col, val)
    new = I.revalue_symmetric(ptr, col, val, seed=3)
    G.partial_rebuild(torch.tensor(new, device="cuda"))
    H.rebuild(new)
    for l in range(H.nlevels):
        assert np.array_equal(G.export_level(l)["A"][2], H.level(l).A.val)
