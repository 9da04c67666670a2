"""Choice between bricks and cell tiles on levels of more than five million cells.

The cycle is the same bit for bit over either form, but a PCG solve is not: its
dot products are summed per block.  So the default solve is bitwise the one of
the forced form it is meant to take and no other: cell tiles where the parts
fill their 32 x 8 columns badly (9 of 32: 0.28), bricks where they fill them
(0.91).  FP64 and FP32 cycles; the default and the forced forms take four cells
a thread on level 0."""
import numpy as np
import pytest

import problems as P

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("parts,ext,bricks", [(600, (9, 32, 32), 0), (1, (180, 180, 180), 1)])
def test_default_form_of_a_large_level(ssamg_lib, parts, ext, bricks, prec):
    S = ssamg_lib
    nx, ny, nz = ext
    n = parts * nx * ny * nz
    assert n > 5_000_000
    coef = [[6.0 + 0.1 * (p % 5)] + [-1.0] * 6 for p in range(parts)]
    b = np.random.default_rng(5).uniform(-1, 1, (1, n))
    prob = P.Problem(3, [((0, 0, 0), (nx - 1, ny - 1, nz - 1))] * parts, P.STENCIL7.copy(), coef,
                     *P._empty_u(), b, name="large")
    _, A = S.matrix_from_problem(prob)
    rhs = torch.as_tensor(b[0], device="cuda")

    def solve(table):
        sv = S.Solver(precision=prec, flexible=prec, coarse_direct=0, tol=1e-8)
        sv.set_tile_table(table)
        sv.setup(A)
        x = torch.zeros_like(rhs)
        assert sv.solve(rhs, x).converged
        return x

    x = solve(None)
    tiles, brick = solve([4] * S.TILE_CLASSES), solve([4 | S.TILE_BRICKS] * S.TILE_CLASSES)
    assert not torch.equal(tiles, brick)  # the two forms can be told apart
    assert torch.equal(x, brick if bricks else tiles)
