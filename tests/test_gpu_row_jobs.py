"""Row jobs of the U part: entry-balanced blocks on levels with long coupling
rows, lanes elsewhere, at the edges of both: rows of one entry, rows longer
than a block's 256 entries, more entries than the 512 slots of a block."""
import numpy as np
import pytest

import problems as P
from oracle import ssamg as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def star(m, length, seed=3):
    """Two m x m x 1 boxes in 3-D; cell (0, 0) of part 0 coupled to `length`
    cells of part 1 and each of those back, the other cells of part 1's first
    row coupled one to one: symmetric, diagonally dominant."""
    rng = np.random.default_rng(seed)
    box = ((0, 0, 0), (m - 1, m - 1, 0))
    rows, n = [], m * m
    diag = [np.full(n, 4.5), np.full(n, 4.5)]
    def link(p, c, q, d, v):
        rows.append((p, c, q, d, v))
        diag[p][c] += abs(v)
    for t in range(length):
        v = -float(rng.uniform(0.1, 1.0))
        link(0, 0, 1, t, v)
        link(1, t, 0, 0, v)
    for t in range(length, min(length + 40, n)):
        v = -float(rng.uniform(0.1, 1.0))
        link(0, t, 1, t, v)
        link(1, t, 0, t, v)
    cell = lambda c: (c % m, c // m, 0)
    coef = [[diag[p].reshape(1, m, m)] + [-1.0] * 4 + [0.0, 0.0] for p in range(2)]
    up, uq = (np.array([r[k] for r in rows], np.int32) for k in (0, 2))
    ui, uj = (np.array([cell(r[k]) for r in rows], np.int32) for k in (1, 3))
    return P.Problem(3, [box, box], P.STENCIL7.copy(), coef, up, ui, np.zeros_like(ui), uq, uj,
                     np.array([r[4] for r in rows]), rng.uniform(-1, 1, (1, 2 * n)), name="star")


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("m,length", [(40, 9), (40, 33), (48, 255), (48, 257), (48, 400)])
def test_cycle_with_long_coupling_rows_matches_oracle(m, length, precision):
    from paper_2205_14273_gb300 import ssamg as S
    prob = star(m, length)
    h = O.setup(prob)
    grid, A = S.matrix_from_problem(prob)
    z = {}
    for tail in (0, 3):
        sv = S.Solver(precision=precision, flexible=precision, use_tail=tail)
        sv.setup(A)
        r = torch.as_tensor(prob.b[0], device="cuda")
        out = torch.zeros_like(r)
        sv.precondition(r, out)
        torch.cuda.synchronize()
        z[tail] = out.cpu().numpy()
    ref = O.vcycle(h, prob.b[0])
    # sums of at most ~1000 products in another order: FP64 1e-12; FP32 rounding
    # times the levels' conditioning 5e-5 (the bounds of the parity tests)
    tol = 1e-12 if precision == 0 else 5e-5
    for out in z.values():
        assert np.abs(out - ref).max() <= tol * np.abs(ref).max()
