"""dL/dg from shared faces: boxes at the edges of its 32 x 8 x 8 blocks, every
order of the seven entries, and coefficients beyond the range of its
reciprocal (those blocks take a division per face)."""
import numpy as np
import pytest

import problems as P
from oracle import ssamg as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 1, 1), (2, 3, 1), (1, 9, 33), (8, 8, 32), (9, 7, 31),
                                   (17, 16, 65), (3, 24, 40), (33, 34, 35), (41, 33, 31),
                                   (70, 9, 65), (257, 13, 11)])
@pytest.mark.parametrize("scale", [1.0, 12.0, 90.0])
def test_gradient_matches_oracle(shape, scale):
    from paper_2205_14273_gb300 import ssamg as S
    rng = np.random.default_rng(5)
    g = rng.normal(size=shape)
    prob = P.diffusion_from_g(g, rng.uniform(-1, 1, g.size))
    order = rng.permutation(7)
    prob.offsets = prob.offsets[order]
    prob.coef = [[prob.coef[0][e] for e in order]]
    _, A = S.matrix_from_problem(prob)
    sv = S.Solver(max_levels=1, coarse_direct=0)
    sv.setup(A)
    gs = scale * g  # the kernel takes g, not the operator's coefficients
    lam, x = rng.uniform(-1, 1, g.size), rng.uniform(-1, 1, g.size)
    dev = [torch.as_tensor(np.ascontiguousarray(v).ravel(), device="cuda") for v in (gs, lam, x)]
    dg = torch.full_like(dev[0], np.nan)
    sv.diffusion_exp_gradient(dev[0], dev[1], dev[2], dg)
    ref = O.diffusion_exp_gradient(gs, lam, x).ravel()
    got = dg.cpu().numpy()
    # six terms, each with the rounding of exp (1 ulp, amplified by k's own
    # factor) and of ~10 operations: 40 ulp of the largest term of the cell
    mag = np.exp(gs.ravel()) * 6 * 4 * 2
    # (where k^2 overflows the formula has no value: NaN on both sides)
    fin = np.isfinite(ref)
    assert np.array_equal(fin, np.isfinite(got))
    assert np.all(np.abs(got - ref)[fin] <= 40 * 2.2e-16 * mag[fin])
