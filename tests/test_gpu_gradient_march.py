"""dL/dg over boxes that the shared-face form marches through several planes at
a time, with ragged edges along every direction, and over boxes that fill its
32 x 8 columns badly (a thread per cell); coefficients beyond the range of its
reciprocal in a few cells, so that whole slabs take a division per face beside
others that do not."""
import numpy as np
import pytest

import problems as P
from oracle import ssamg as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def planes(shape):
    """Planes a block of the shared-face form marches; 0: a thread per cell."""
    nz, ny, nx = shape
    cols = -(-nx // 32) * -(-ny // 8)
    if nz * ny * nx < 152 * 256 or nz * ny * nx < 0.47 * cols * 256 * nz:
        return 0
    return max(1, min(8, cols * nz // (4 * 152)))


@pytest.mark.parametrize("shape,march", [((61, 64, 65), 2), ((83, 67, 70), 3), ((84, 80, 97), 5),
                                         ((131, 101, 97), 8), ((129, 96, 128), 8),
                                         ((300, 9, 33), 0), ((700, 2, 64), 0), ((34, 34, 34), 0),
                                         ((60, 100, 16), 1), ((1, 400, 400), 1)])
@pytest.mark.parametrize("far", [False, True])
def test_gradient_matches_oracle(shape, march, far):
    from paper_2205_14273_gb300 import ssamg as S
    assert planes(shape) == march
    rng = np.random.default_rng(11)
    g = rng.normal(size=shape)
    prob = P.diffusion_from_g(g, np.zeros(g.size))
    _, A = S.matrix_from_problem(prob)
    sv = S.Solver(max_levels=1, coarse_direct=0)
    sv.setup(A)
    if far:
        # (k_c + k_n)^2 of 2^231 beside one face of a block, inside and at a corner
        for c in ((0, 0, 0), (shape[0] // 2, shape[1] // 2, min(32, shape[2] - 1)),
                  (shape[0] - 1, shape[1] - 1, shape[2] // 3)):
            g[c] = 80.0
    lam, x = rng.uniform(-1, 1, g.size), rng.uniform(-1, 1, g.size)
    dev = [torch.as_tensor(np.ascontiguousarray(v).ravel(), device="cuda") for v in (g, lam, x)]
    dg = torch.full_like(dev[0], np.nan)
    sv.diffusion_exp_gradient(dev[0], dev[1], dev[2], dg)
    ref = O.diffusion_exp_gradient(g, lam, x).ravel()
    # six terms of at most 2 x 2 x 2 k each, the rounding of exp (1 ulp, amplified by
    # k's own factor) and of ~10 operations: 40 ulp of the cell's largest sum
    assert np.all(np.abs(dg.cpu().numpy() - ref) <= 40 * 2.2e-16 * np.exp(g.ravel()) * 48)
