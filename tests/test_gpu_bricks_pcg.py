"""Brick forms of the PCG's own kernels and of the caller's apply, on ragged
parts and several problems: forced by the tile table where the built-in rule
would keep cell tiles, and the regime where the rule takes bricks in the FP32
cycle and cell tiles in the FP64 applies."""
import numpy as np
import pytest

import problems as P
from oracle import ssamg as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu



def columns(n):
    """Couplings along x per cell, constants along y and z."""
    rng = np.random.default_rng(8)
    t = np.zeros((n, n, n + 1))
    t[:, :, 1:-1] = rng.uniform(0.5, 20.0, (n, n, n - 1))
    prob = P.laplace7(n)
    prob.coef = [[t[:, :, 1:] + t[:, :, :-1] + 4.01, -t[:, :, :-1], -t[:, :, 1:], -1.0, -1.0, -1.0, -1.0]]
    prob.name = f"columns {n}^3"
    return prob


# (stencils whose entries are not all per cell: the levels that bricks are for)
CASES = [P.laplace7(33), P.multipart_aniso(m=13, layout=(2, 1, 2), seed=3), P.samr(20), columns(19),
         P.laplace7(5)]


def table(S):
    return [1 | S.TILE_BRICKS] * S.TILE_CLASSES


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("prob", CASES, ids=[p.name for p in CASES])
def test_forced_bricks_match_cell_tiles(prob, precision):
    from paper_2205_14273_gb300 import ssamg as S
    _, A = S.matrix_from_problem(prob)
    rng = np.random.default_rng(3)
    r = torch.as_tensor(rng.uniform(-1, 1, prob.n), device="cuda")
    b = torch.as_tensor(prob.b[0], device="cuda")
    out = []
    for bricks in (0, 1):
        sv = S.Solver(precision=precision, flexible=precision, use_bricks=bricks, tol=1e-12,
                      max_iter=500)
        sv.set_tile_table(table(S) if bricks else None)
        sv.setup(A)
        assert sv.level_tile(0)[1] == bricks
        z, y, x = (torch.zeros_like(r) for _ in range(3))
        sv.precondition(r, z)
        sv.level_matvec(0, r, y)
        st = sv.solve(b, x)
        assert st.converged and st.true_rel_res <= 1e-11
        out.append((z, y, x, st.iterations))
    # a cell's sum runs in one order in both forms; the dot products do not
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    assert abs(out[0][3] - out[1][3]) <= 1
    assert float((out[0][2] - out[1][2]).abs().max()) <= 1e-9 * float(out[0][2].abs().max())
    ref = O.matvec(O.level0_from_problem(prob), r.cpu().numpy())
    assert np.abs(out[1][1].cpu().numpy() - ref).max() <= 1e-13 * np.abs(ref).max()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("together", [0, 1])
def test_forced_bricks_in_a_batch(precision, together):
    """Per-problem ranges of the brick partials, several right-hand sides."""
    from paper_2205_14273_gb300 import ssamg as S
    probs = P.batched(nprob=5, nrhs=3, seed=17, pmax=3, emin=4, emax=19)
    mats = [S.matrix_from_problem(p)[1] for p in probs]
    res = []
    for bricks in (0, 1):
        B = S.Batch(mats, precision=precision, flexible=precision, use_bricks=bricks, tol=1e-12,
                    max_iter=500, rhs_together=together)
        B.solver().set_tile_table(table(S) if bricks else None)
        B.setup()
        assert B.solver().level_tile(0)[1] == bricks
        b = torch.as_tensor(np.stack([np.concatenate([p.b[j] for p in probs]) for j in range(3)]),
                            device="cuda")
        x = torch.zeros_like(b)
        st = B.solve(b, x, 3)
        res.append((x, [[s.iterations for s in row] for row in st]))
        assert all(s.converged and s.true_rel_res <= 1e-11 for row in st for s in row)
    assert np.abs(np.array(res[0][1]) - np.array(res[1][1])).max() <= 1
    assert float((res[0][0] - res[1][0]).abs().max()) <= 1e-9 * float(res[0][0].abs().max())


@pytest.mark.parametrize("together", [0, 1])
def test_fp32_cycle_over_bricks_fp64_applies_over_tiles(together):
    """66^3, 61^3 and 70^3: 614 bricks, 0.68 full, so above the rule's line for
    FP32 (250, 0.6) and below its line for FP64 (800, 0.85)."""
    from paper_2205_14273_gb300 import ssamg as S
    probs = [P.laplace7(n, nrhs=2, seed=n) for n in (66, 61, 70)]
    mats = [S.matrix_from_problem(p)[1] for p in probs]
    res = []
    for bricks in (0, 1):
        B = S.Batch(mats, precision=1, flexible=1, use_bricks=bricks, tol=1e-12, max_iter=500,
                    rhs_together=together)
        B.setup()
        b = torch.as_tensor(np.stack([np.concatenate([p.b[j] for p in probs]) for j in range(2)]),
                            device="cuda")
        x = torch.zeros_like(b)
        st = B.solve(b, x, 2)
        res.append((x, [[s.iterations for s in row] for row in st]))
        assert all(s.converged and s.true_rel_res <= 1e-11 for row in st for s in row)
    assert np.abs(np.array(res[0][1]) - np.array(res[1][1])).max() <= 1
    assert float((res[0][0] - res[1][0]).abs().max()) <= 1e-9 * float(res[0][0].abs().max())
