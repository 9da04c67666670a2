"""Entry-balanced row jobs whose block holds more entries than its 512 slots:
short rows first and then a row of hundreds of entries that starts in the same
block, on level 0 and on the level below it; those blocks go back to lanes."""
import numpy as np
import pytest

import problems as P
from oracle import ssamg as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ENTRIES, SLOTS = 256, 512


def late_hub(m, short, length, step, seed=3):
    """Two m x m x 1 boxes in 3-D; the first `short` cells of part 0 coupled one to
    one to cells of part 1, the next cell (the hub) to `length` cells of part 1,
    and each of those back: symmetric, diagonally dominant.  Cells are `step`
    apart: with 2 they are coarse points, whose rows keep their lengths."""
    rng = np.random.default_rng(seed)
    box = ((0, 0, 0), (m - 1, m - 1, 0))
    n = m * m
    diag = [np.full(n, 4.5), np.full(n, 4.5)]
    rows = []
    pairs = [(t, length + t) for t in range(short)] + [(short, t) for t in range(length)]
    for c, d in pairs:
        c, d = step * c, step * d
        v = -float(rng.uniform(0.1, 1.0))
        rows += [(0, c, 1, d, v), (1, d, 0, c, v)]
        diag[0][c] += abs(v)
        diag[1][d] += abs(v)
    cell = lambda c: (c % m, c // m, 0)
    coef = [[diag[p].reshape(1, m, m)] + [-1.0] * 4 + [0.0, 0.0] for p in range(2)]
    up, uq = (np.array([r[k] for r in rows], np.int32) for k in (0, 2))
    ui, uj = (np.array([cell(r[k]) for r in rows], np.int32) for k in (1, 3))
    return P.Problem(3, [box, box], P.STENCIL7.copy(), coef, up, ui, np.zeros_like(ui), uq, uj,
                     np.array([r[4] for r in rows]), rng.uniform(-1, 1, (1, 2 * n)), name="late hub")


def most_entries(lev):
    """Most entries of a block: rows whose entries start in a window of ENTRIES."""
    cells, counts = np.unique(lev.u_row, return_counts=True)
    ptr = np.concatenate([[0], np.cumsum(counts)])
    best = 0
    for k in range(-(-int(ptr[-1]) // ENTRIES)):
        r = np.searchsorted(ptr[:-1], [k * ENTRIES, (k + 1) * ENTRIES])
        best = max(best, int(ptr[r[1]] - ptr[r[0]]))
    return best


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("short,length,step", [(240, 273, 1), (240, 400, 1), (250, 262, 1),
                                               (100, 400, 1), (240, 273, 2), (250, 400, 2)])
def test_cycle_and_solve_match_oracle(short, length, step, precision):
    from paper_2205_14273_gb300 import ssamg as S
    prob = late_hub(48, short, length, step)
    h = O.setup(prob)
    assert most_entries(h.levels[0]) == short + length
    assert step == 1 or most_entries(h.levels[1]) > SLOTS
    _, A = S.matrix_from_problem(prob)
    sv = S.Solver(precision=precision, flexible=precision, use_tail=0, tol=1e-12)
    sv.setup(A)
    r = torch.as_tensor(prob.b[0], device="cuda")
    z, x = torch.zeros_like(r), torch.zeros_like(r)
    sv.precondition(r, z)
    st = sv.solve(r, x)
    ref = O.vcycle(h, prob.b[0])
    pcg = O.pcg(h, prob.b[0], tol=1e-12)
    # sums of at most ~1000 products in another order: FP64 1e-12; FP32 rounding
    # times the levels' conditioning 5e-5 (the bounds of the parity tests)
    tol = 1e-12 if precision == 0 else 5e-5
    assert np.abs(z.cpu().numpy() - ref).max() <= tol * np.abs(ref).max()
    assert st.converged and abs(st.iterations - pcg.iterations) <= 1
    assert np.abs(x.cpu().numpy() - pcg.x).max() <= 1e-10 * np.abs(pcg.x).max()
