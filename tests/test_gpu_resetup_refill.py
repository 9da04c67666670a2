"""One Matrix refilled and assembled again, one Solver set up again, as a time
step does: where the matrix's arrays come back at the same addresses (no
couplings, so each of its sizes is freed and taken once, and nothing else is in
the cache) the instantiated solve graphs stay and must serve the new operator; what the launches depend on beside the values
(tile table, couplings, right-hand sides, their buffers, coarsening) must
give new ones.  Every solution bitwise a fresh solver's."""
import numpy as np
import pytest

import problems as P

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

MAXR = 5
# couplings along x, y, z: other values under the same coarsening, and another one
STEPS = [(1, 1, 1), (3, 3, 3), (0.5, 0.5, 0.5), (40, 1, 1), (50, 1, 1), (60, 1, 1), (1, 1, 40),
         (1, 1, 30), (2, 2, 2), (1, 1, 1), (1, 1, 1)]
TABLE, SPACINGS = 9, 10  # the steps with a tile table and with given spacings


def refill(S, A, prob):
    for e, c in enumerate(prob.coef[0]):
        if np.isscalar(c):
            A.set_constant(0, e, float(c))
        else:
            A.set_box_values(0, e, torch.as_tensor(np.ascontiguousarray(c).ravel(), device="cuda"))
    A.assemble()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("varying", [False, True])
@pytest.mark.parametrize("rounds,together", [((1, 3, 1), 0), ((1, 3, 1), 1), ((5, 3, 1, 5), 1)])
def test_refilled_matrix_under_kept_graphs(precision, varying, rounds, together):
    from paper_2205_14273_gb300 import ssamg as S
    S.lib().ssamg_release_device_cache()
    n = 21
    rng = np.random.default_rng(6)

    def problem(step):
        prob = P.laplace7(n, nrhs=MAXR, seed=step)
        ax, ay, az = STEPS[step]
        d = 2.0 * (ax + ay + az) + 0.01
        diag = rng.uniform(d, 1.2 * d, (n, n, n)) if varying else d
        prob.coef = [[diag, -ax, -ax, -ay, -ay, -az, -az]]
        return prob

    prob = problem(0)
    grid, A = S.matrix_from_problem(prob)
    kw = dict(precision=precision, flexible=precision, rhs_together=together)
    sv = S.Solver(**kw)
    bs = torch.empty((MAXR, prob.n), dtype=torch.float64, device="cuda")
    xs = torch.empty_like(bs)
    alive = []  # (the fresh objects' arrays do not enter the cache)
    for step in range(len(STEPS)):
        prob = problem(step)
        refill(S, A, prob)
        _, A2 = S.matrix_from_problem(prob)
        fresh = S.Solver(**kw)
        alive.append((fresh, A2))
        for s in (sv, fresh):
            s.set_tile_table([2] * S.TILE_CLASSES if step == TABLE else None)
            s.set_spacings([[1.0, 2.0, 4.0]] if step == SPACINGS else None)
        sv.setup(A)
        fresh.setup(A2)
        bs.copy_(torch.as_tensor(prob.b, device="cuda"))
        for nrhs in rounds:  # the same buffers in every step
            xs.zero_()
            y = torch.zeros_like(xs)
            s1, s2 = sv.solve(bs, xs, nrhs), fresh.solve(bs, y, nrhs)
            assert s1.converged and s1.iterations == s2.iterations, (step, nrhs)
            assert torch.equal(xs, y), (step, nrhs)


@pytest.mark.parametrize("precision", [0, 1])
def test_one_matrix_set_up_again_and_again(precision):
    """The same coupled matrix, unchanged: the graph stays between the set-ups;
    another matrix and another table in between give their own."""
    from paper_2205_14273_gb300 import ssamg as S
    prob = P.multipart_aniso(m=13, layout=(2, 1, 2), seed=3, nrhs=3)
    other = P.multipart_aniso(m=13, layout=(2, 1, 2), seed=9, nrhs=3)
    mats = [S.matrix_from_problem(p)[1] for p in (prob, other)]
    kw = dict(precision=precision, flexible=precision)
    sv = S.Solver(**kw)
    b = torch.as_tensor(prob.b.copy(), device="cuda")
    x = torch.zeros_like(b)
    ref = {}
    for m, tab in ((0, 0), (0, 0), (1, 0), (0, 0), (0, 3), (0, 3), (0, 0), (1, 0), (1, 3), (0, 0)):
        sv.set_tile_table([tab] * S.TILE_CLASSES if tab else None)
        sv.setup(mats[m])
        if (m, tab) not in ref:
            fresh = S.Solver(**kw)
            fresh.set_tile_table([tab] * S.TILE_CLASSES if tab else None)
            fresh.setup(mats[m])
            y = {n: torch.zeros_like(b) for n in (1, 3)}
            for n in y:
                fresh.solve(b, y[n], n)
            ref[m, tab] = y
        for n in (1, 3):
            x.zero_()
            sv.solve(b, x, n)
            assert torch.equal(x, ref[m, tab][n]), (m, tab, n)
