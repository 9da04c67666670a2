"""A batch without the direct coarsest solve keeps its problems apart: a NaN in
one problem's right-hand side leaves the others' solutions as they are, bit for
bit, also where the small levels of the FP64 cycle are folded into one matrix
for a single problem."""
import numpy as np
import pytest

import problems as P

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("bad", [1, 2])
def test_a_nan_stays_in_its_problem(precision, bad):
    from paper_2205_14273_gb300 import ssamg as S
    probs = [P.laplace7(9), P.laplace7(12), P.laplace7(11)]
    mats = [S.matrix_from_problem(p)[1] for p in probs]
    B = S.Batch(mats, precision=precision, flexible=precision, coarse_direct=0)
    B.setup()
    off = B.offsets()
    b = np.concatenate([p.b[0] for p in probs])
    x = [torch.zeros(off[-1], dtype=torch.float64, device="cuda") for _ in range(2)]
    st = B.solve(torch.as_tensor(b, device="cuda"), x[0], 1)
    assert all(s.converged for s in st[0])
    b[off[bad] + 5] = np.nan
    with pytest.raises(S.SsamgError):
        B.solve(torch.as_tensor(b, device="cuda"), x[1], 1)
    for k in range(3):
        if k != bad:
            assert torch.equal(x[0][off[k]:off[k + 1]], x[1][off[k]:off[k + 1]]), k
