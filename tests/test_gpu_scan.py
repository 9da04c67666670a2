"""Coupling sums over hierarchies whose coupling-row counts cross the sizes of
the scan's forms (one block of up to 16384 items; blocks of 1024 beyond)."""
import pytest

import problems as P
from oracle import ssamg as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,layout", [(3, (2, 1, 1)), (16, (2, 2, 1)), (32, (2, 1, 1)),
                                      (26, (2, 2, 2)), (41, (2, 2, 1))])
def test_coupling_rows_match_oracle(m, layout):
    import numpy as np
    from paper_2205_14273_gb300 import ssamg as S
    prob = P.multipart_aniso(m=m, layout=layout, seed=4)
    h = O.setup(prob)
    _, A = S.matrix_from_problem(prob)
    sv = S.Solver()
    sv.setup(A)
    assert sv.num_levels() == len(h.levels)
    for l in range(sv.num_levels()):
        n, nr, nnz = sv.level_sizes(l)
        ptr = sv.level_copy(l, 4, n=nr + 1, dtype=np.int32) if nr else np.zeros(1, np.int32)
        rows = sv.level_copy(l, 5, n=nr, dtype=np.int32) if nr else np.zeros(0, np.int32)
        col = sv.level_copy(l, 6, n=nnz, dtype=np.int32) if nnz else np.zeros(0, np.int32)
        assert ptr[0] == 0 and ptr[-1] == nnz and (np.diff(ptr) >= 0).all()
        assert (np.diff(rows) > 0).all() and (col < n).all()
        got = {(int(r), int(c)) for i, r in enumerate(rows) for c in col[ptr[i]:ptr[i + 1]]}
        lev = h.levels[l]
        assert got == set(zip(lev.u_row.tolist(), lev.u_col.tolist())), l
