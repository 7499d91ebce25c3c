"""A caller's pattern that is wrong is reported as such whatever form its
columns would be stored in: by diagonals (up to eight offsets), one byte or two
bytes an entry, int32."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from paper_2108_02054_gb300 import amg as B

N = 600


def banded(half, fault):
    """Rows of the columns i - half .. i + half, the row in the middle wrong."""
    rows = [list(range(max(0, i - half), min(N, i + half + 1))) for i in range(N)]
    r = rows[N // 2]
    if fault == "twice":
        r[1] = r[0]
    elif fault == "unsorted":
        r[0], r[1] = r[1], r[0]
    elif fault == "no diagonal":
        r.remove(N // 2)
    elif fault == "out of range":
        r[-1] = N + half
    ptr = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int32)
    col = np.concatenate(rows).astype(np.int32)
    val = np.where(col == np.repeat(np.arange(N), np.diff(ptr)), 2.0 * half + 0.5, -1.0)
    return [torch.tensor(a, device="cuda") for a in (ptr, col, val)]


@pytest.mark.parametrize("half", [1, 3, 4, 140])
@pytest.mark.parametrize("fault", ["twice", "unsorted", "no diagonal", "out of range"])
@pytest.mark.parametrize("entry", ["full_setup", "step"])
def test_wrong_rows(half, fault, entry):
    G = B.AMG()
    good = banded(half, None)
    G.full_setup(*good)
    ptr, col, val = banded(half, fault)
    with pytest.raises(B.AmgError) as e:
        if entry == "step":
            G = B.AMG()
            G.step(val, ptr, col)
        else:
            G.full_setup(ptr, col, val)
    assert e.value.status == B.AMG_ERR_PATTERN, str(e.value)
    with pytest.raises(B.AmgError) as e:  # no hierarchy is left
        G.partial_rebuild(val)
    assert e.value.status == B.AMG_ERR_STATE
    G.full_setup(*good)
    f = torch.ones(N, dtype=torch.float64, device="cuda")
    assert G.solve(f, 1e-8)[1].status == 0
