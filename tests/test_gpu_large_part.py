"""A 27-point part whose entry-major coefficients pass 2^31 elements: 437^3
cells, so that entry 26 starts at element 26 x 83,453,453 = 2,169,789,778.
The caller's apply and the apply of a PCG step against the same sums formed
by slices."""
import numpy as np
import pytest

import problems as P

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.slow]

M = 437


def test_applies_of_a_part_with_more_than_2_31_coefficients():
    from paper_2205_14273_gb300 import ssamg as S
    assert 26 * M ** 3 > 2 ** 31
    if torch.cuda.mem_get_info()[0] < 80e9:
        pytest.skip("needs 80 GB of device memory")
    offs = [(i, j, k) for k in (-1, 0, 1) for j in (-1, 0, 1) for i in (-1, 0, 1)]
    # a value per pair (o, -o), so that the operator is symmetric and every
    # pair tells itself from the others
    w = {o: (30.0 if o == (0, 0, 0) else -(0.2 + 0.05 * min(e, 26 - e))) for e, o in enumerate(offs)}
    grid = S.Grid(3, [((0, 0, 0), (M - 1,) * 3)])
    A = S.Matrix(grid, np.array(offs, np.int32))
    fill = torch.empty(M ** 3, dtype=torch.float64, device="cuda")
    for e, o in enumerate(offs):
        A.set_box_values(0, e, fill.fill_(w[o]))
    A.assemble()
    sv = S.Solver(max_levels=1, coarse_direct=0, max_iter=1, tol=0.0)
    sv.setup(A)
    gen = torch.Generator(device="cuda").manual_seed(3)
    x = torch.rand(M, M, M, dtype=torch.float64, device="cuda", generator=gen) * 2 - 1

    def apply(v):
        p = torch.nn.functional.pad(v, (1,) * 6)
        y = torch.zeros_like(v)
        for i, j, k in offs:
            y += w[i, j, k] * p[1 + k:M + 1 + k, 1 + j:M + 1 + j, 1 + i:M + 1 + i]
        return y

    y = torch.empty_like(x)
    sv.level_matvec(0, x, y)
    ref = apply(x)
    # 27 products each way, in another order
    assert float((y - ref).abs().max()) <= 2 * 27 * 2.3e-16 * sum(abs(v) for v in w.values())
    # one PCG step from zero: z = D b, x1 = (b.z / z.Az) z
    b, x1 = x, torch.zeros_like(x)
    sv.solve(b, x1, allow_not_converged=True)
    z = b * (sv.part_info(0, 0)["omega"] / w[0, 0, 0])
    want = z * ((b * z).sum() / (z * apply(z)).sum())
    # sums of 8e7 terms of one sign or decaying as their root: 1e-11 of their size
    assert float((x1 - want).abs().max()) <= 1e-11 * float(want.abs().max())
