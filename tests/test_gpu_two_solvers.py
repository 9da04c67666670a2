"""Two live solvers whose coarse-level transitions need different amounts of
shared memory: setting the smaller one up must not stop the larger one."""
import pytest

import problems as P

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
def test_a_smaller_transition_set_up_later(precision):
    from paper_2205_14273_gb300 import ssamg as S
    out = []
    probs = [P.multipart_aniso(m=24, layout=(2, 2, 2), seed=3), P.laplace7(16)]
    mats = [S.matrix_from_problem(p)[1] for p in probs]
    kw = dict(precision=precision, flexible=precision)
    b = torch.as_tensor(probs[0].b[0], device="cuda")
    for later in (False, True):
        big = S.Solver(**kw)
        big.setup(mats[0])
        if later:
            small = S.Solver(tail_cells=512, **kw)
            small.setup(mats[1])
        z = torch.zeros_like(b)
        big.precondition(b, z)
        x = torch.zeros_like(b)
        big.solve(b, x)
        out.append((z, x))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
