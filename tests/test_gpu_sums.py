"""The coupling sums (Section 3.1) do not depend on the tile table: a
partition that followed it rounded them, and with them omega and the cycle,
differently (seen on this problem with 3 cells per thread)."""
import pytest

import problems as P

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_sums_and_cycle_are_the_same_under_every_tile_table():
    from paper_2205_14273_gb300 import ssamg as S
    prob = P.multipart_aniso(m=13, layout=(2, 2, 1), seed=1)
    _, A = S.matrix_from_problem(prob)
    r = torch.as_tensor(P.SplitMix64(17).uniform_pm1(prob.n), device="cuda")
    ref = None
    for t in (None, 1, 2, 3, 4):
        sv = S.Solver()
        sv.set_tile_table(None if t is None else [t] * S.TILE_CLASSES)
        sv.setup(A)
        z = torch.zeros_like(r)
        sv.precondition(r, z)
        c, W = sv.spacings()
        if ref is None:
            ref = (z, c, W)
        assert (c == ref[1]).all() and (W == ref[2]).all() and torch.equal(z, ref[0]), t
