"""A solver set up again: the solve graph kept over set-ups of the same shape
serves the new operator, and another shape, precision of tiles or number of
right-hand sides gets its own, all bitwise a fresh solver's results."""
import pytest

import problems as P

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
def test_set_up_again_solves_the_new_operator(precision):
    from paper_2205_14273_gb300 import ssamg as S
    probs = [P.multipart_aniso(m=13, layout=(2, 1, 2), seed=3, nrhs=3),
             P.multipart_aniso(m=13, layout=(2, 1, 2), seed=3, nrhs=3),   # the same shape
             P.multipart_aniso(m=13, layout=(2, 1, 2), seed=9, nrhs=3),   # other directions
             P.laplace7(20, nrhs=3), P.laplace7(20, nrhs=3), P.laplace7(21, nrhs=3)]
    probs[1].coef = [[2.0 * c for c in part] for part in probs[1].coef]
    probs[1].u_val = 2.0 * probs[1].u_val
    probs[4].coef = [[0.5 * c for c in part] for part in probs[4].coef]
    sv = S.Solver(precision=precision, flexible=precision)
    mats = [S.matrix_from_problem(p)[1] for p in probs]
    for step, (prob, A) in enumerate(zip(probs, mats)):
        fresh = S.Solver(precision=precision, flexible=precision)
        sv.set_tile_table([2] * S.TILE_CLASSES if step == 5 else None)
        fresh.set_tile_table([2] * S.TILE_CLASSES if step == 5 else None)
        sv.setup(A)
        fresh.setup(A)
        for nrhs in (1, 3, 1, 2):
            b = torch.as_tensor(prob.b[:nrhs].copy(), device="cuda")
            x, y = torch.zeros_like(b), torch.zeros_like(b)
            s1, s2 = sv.solve(b, x, nrhs), fresh.solve(b, y, nrhs)
            assert s1.iterations == s2.iterations and torch.equal(x, y), (step, nrhs)
