"""The work a program has this library do, as cases that can be timed.

A case names a kind of system (how parts, coefficients and couplings are
laid out), its sizes, and what is asked of the library:

  step       the hierarchy of a new operator and one PCG solve: what an
             implicit time step or a nonlinear iteration does
  solve      PCG solves on a hierarchy that is kept (one operator, given by
             the case's "op", and right-hand sides that change)
  batch      hierarchy and solves of many small independent systems at once
  train      forward and backward through the differentiable solve: grid,
             matrix and hierarchy from a coefficient tensor, forward solve,
             adjoint solve, gradients of the coefficients and of b
  gradient   dL/dg of the exp-diffusion operator for a given adjoint
  cycle      one V(1,1) cycle as the preconditioner of a caller's own Krylov
             loop (the operator again given by "op")
  apply      y = A x with the assembled operator (a caller's residuals)

Kinds of system (sizes in cells):

  grid       lx x ly x lz equal parts of nx x ny x nz cells, constant
             anisotropic off-diagonals per part, harmonic couplings between
             facing parts, Dirichlet elsewhere (2-D with nz = 0)
  chain      cube parts of the given edges in a row along x, coupled on the
             overlap of facing sides: uneven parts, partly coupled faces
  var27      one part n^3, 27-point operator, coefficients constant on 8^3
             blocks over eight decades
  samr       a coarse part m^3 with ghost unknowns under a patch refined by
             two (m^3 cells), coupled across the patch's faces
  diffusion  one part n^3, 7-point harmonic diffusion with kappa = exp(g),
             g smoothed noise
"""
import numpy as np
import torch

from paper_2205_14273_gb300 import autograd as AD
from paper_2205_14273_gb300 import ssamg as S

P5 = [(0, 0, 0), (-1, 0, 0), (1, 0, 0), (0, -1, 0), (0, 1, 0)]
P7 = P5 + [(0, 0, -1), (0, 0, 1)]
P27 = [(0, 0, 0)] + [(i, j, k) for k in (-1, 0, 1) for j in (-1, 0, 1) for i in (-1, 0, 1)
                     if (i, j, k) != (0, 0, 0)]
EXACT_CELLS = 4_500_000  # largest system whose exact solution is computed


def listed():
    return [
        # the smallest calls: one 32^3 box, Laplacian, everything default; a
        # user's first program, and the inner solve of a larger scheme
        {"name": "laplace_32", "do": "step", "kind": "grid", "lx": 1, "ly": 1, "lz": 1,
         "nx": 32, "ny": 32, "nz": 32, "iso": True, "precision": 0},
        # the benchmark's workload: eight anisotropic 64^3 parts, FP32 cycle
        {"name": "aniso_8x64_f32", "do": "step", "kind": "grid", "lx": 2, "ly": 2, "lz": 2,
         "nx": 64, "ny": 64, "nz": 64, "iso": False, "precision": 1},
        # the same parts with the default FP64 cycle, the hierarchy kept over
        # many right-hand sides (implicit time stepping with a fixed operator)
        {"name": "aniso_8x64_f64", "do": "solve", "kind": "grid", "lx": 2, "ly": 2, "lz": 2,
         "nx": 64, "ny": 64, "nz": 64, "iso": False, "precision": 0, "nrhs": 1, "op": 1},
        # uneven parts of odd sizes in a row, FP32 cycle
        {"name": "chain_ragged_f32", "do": "step", "kind": "chain", "edges": "96,37,61,83,23",
         "precision": 1},
        # the largest: 16.8M unknowns, 27-point, coefficients over 8 decades
        {"name": "var27_256_f32", "do": "step", "kind": "var27", "n": 256, "precision": 1},
        # a 2-D plane of four odd-sized parts, FP64
        {"name": "plane_4x511", "do": "step", "kind": "grid", "lx": 2, "ly": 2, "lz": 1,
         "nx": 511, "ny": 509, "nz": 0, "iso": False, "precision": 0},
        # adaptive refinement: ghost unknowns, couplings inside a part; one
        # operator, several right-hand sides
        {"name": "samr_96_f32", "do": "solve", "kind": "samr", "m": 96, "precision": 1, "nrhs": 2,
         "op": 1},
        # many uneven problems with several right-hand sides each
        {"name": "batch_12x4_f32", "do": "batch", "kind": "batch", "nprob": 12, "nrhs": 4,
         "emin": 16, "emax": 64, "precision": 1, "op": 1},
        # a training step through the solve (coefficients as parameters)
        {"name": "train_96", "do": "train", "kind": "diffusion", "n": 96},
        # the gradient kernel of the exp parametrisation on the 128^3 box
        {"name": "gradient_128", "do": "gradient", "kind": "diffusion", "n": 128},
        # one cycle inside a caller's Krylov method
        {"name": "cycle_8x64_f32", "do": "cycle", "kind": "grid", "lx": 2, "ly": 2, "lz": 2,
         "nx": 64, "ny": 64, "nz": 64, "iso": False, "precision": 1, "op": 1},
        # operator apply on the same parts
        {"name": "apply_8x64", "do": "apply", "kind": "grid", "lx": 2, "ly": 2, "lz": 2,
         "nx": 64, "ny": 64, "nz": 64, "iso": False, "precision": 0},
    ]


def _log(rng, a, b):
    return int(round(a * (b / a) ** rng.random()))


def draw(rng):
    do = rng.choice(["step", "step", "step", "solve", "solve", "batch", "train", "gradient",
                     "cycle", "apply"])
    if do == "batch":
        emin = _log(rng, 8, 32)
        c = {"do": do, "kind": "batch", "nprob": _log(rng, 2, 16), "nrhs": rng.randint(1, 4),
             "emin": emin, "emax": emin + _log(rng, 8, 64), "precision": rng.randint(0, 1),
             "op": rng.randint(1, 999)}
        while c["nprob"] > 2 and _unknowns(c) * c["nrhs"] > 8_000_000:
            c["nprob"] -= 1
        return c
    if do == "train":
        return {"do": do, "kind": "diffusion", "n": _log(rng, 12, 112)}
    if do == "gradient":
        return {"do": do, "kind": "diffusion", "n": _log(rng, 16, 224)}
    kind = rng.choice(["grid", "grid", "plane", "chain", "var27", "samr"])
    c = {"do": do, "kind": kind, "precision": rng.randint(0, 1)}
    if do == "solve":
        c["nrhs"] = rng.randint(1, 4)
    if do in ("solve", "cycle"):
        c["op"] = rng.randint(1, 999)
    if kind == "grid":
        lx, ly, lz = rng.choice([(1, 1, 1), (2, 1, 1), (2, 2, 1), (2, 2, 2), (3, 2, 1)])
        n = _log(rng, 9, 96)
        c.update(lx=lx, ly=ly, lz=lz, nx=n, ny=max(3, n - rng.randint(0, n // 3)),
                 nz=max(3, n - rng.randint(0, n // 3)), iso=rng.random() < 0.25)
    elif kind == "plane":
        lx, ly = rng.choice([(1, 1), (2, 1), (2, 2), (3, 2)])
        n = _log(rng, 24, 900)
        c.update(kind="grid", lx=lx, ly=ly, lz=1, nx=n, ny=max(9, n - rng.randint(0, n // 3)),
                 nz=0, iso=rng.random() < 0.25)
    elif kind == "chain":
        hi = _log(rng, 16, 96)
        c["edges"] = ",".join(str(rng.randint(max(5, hi // 4), hi))
                              for _ in range(rng.randint(2, 6)))
    elif kind == "var27":
        c["n"] = _log(rng, 16, 160)
    else:
        c["m"] = 4 * _log(rng, 3, 28)
    while c.get("nrhs", 1) > 1 and _unknowns(c) * c["nrhs"] > 3_500_000:
        c["nrhs"] -= 1
    return c


def _unknowns(c):
    if c["kind"] == "batch":
        return sum(v ** 3 for e in _batch_edges(c) for v in e)
    if c["kind"] == "grid":
        return c["lx"] * c["ly"] * c["lz"] * c["nx"] * c["ny"] * max(1, c["nz"])
    if c["kind"] == "chain":
        return sum(int(v) ** 3 for v in c["edges"].split(","))
    return c["n"] ** 3 if "n" in c else 2 * c["m"] ** 3


# ------------------------------------------------------------ systems ------
def _uniform(n, gen, lo=-1.0, hi=1.0):
    return torch.rand(n, dtype=torch.float64, device="cuda", generator=gen) * (hi - lo) + lo


def _harm(a, b):
    return 2.0 * a * b / (a + b)


def _aniso(host, iso):
    return np.ones(3) if iso else np.exp(host.uniform(np.log(1e-3), 0.0, 3))


class _Links:
    """Couplings in the form Matrix.add_couplings takes."""

    def __init__(self):
        self.rows = []

    def add(self, p, cells, direction, q, nbors, value):
        self.rows.append((np.full(len(cells), p, np.int32), cells,
                          np.tile(np.asarray(direction, np.int32), (len(cells), 1)),
                          np.full(len(cells), q, np.int32), nbors,
                          np.full(len(cells), float(value))))

    def arrays(self):
        if not self.rows:
            return None
        out = [np.concatenate(c) for c in zip(*self.rows)]
        return tuple(np.ascontiguousarray(a, np.float64 if i == 5 else np.int32)
                     for i, a in enumerate(out))


def _system(ndim, offsets, boxes, coef, links):
    return {"ndim": ndim, "offsets": offsets, "boxes": boxes, "coef": coef,
            "links": links.arrays()}


def _grid(c, host):
    """Parts in a block layout; coefficients per part (a_x, a_y, a_z)."""
    flat = c["nz"] == 0
    n = (c["nx"], c["ny"], max(1, c["nz"]))
    lay = (c["lx"], c["ly"], c["lz"])
    ndim = 2 if flat else 3
    npart = lay[0] * lay[1] * lay[2]
    a = np.stack([_aniso(host, c["iso"]) for _ in range(npart)])
    links, coef = _Links(), []
    for p in range(npart):
        pos = (p % lay[0], (p // lay[0]) % lay[1], p // (lay[0] * lay[1]))
        diag = torch.full((n[2], n[1], n[0]), 2.0 * float(a[p, :ndim].sum()),
                          dtype=torch.float64, device="cuda")
        for d in range(ndim):
            for s in (-1, 1):
                nb = list(pos)
                nb[d] += s
                if not 0 <= nb[d] < lay[d]:
                    continue
                q = nb[0] + lay[0] * (nb[1] + lay[1] * nb[2])
                u = -_harm(a[p, d], a[q, d])
                face = n[d] - 1 if s > 0 else 0
                sl = [slice(None)] * 3
                sl[2 - d] = face
                diag[tuple(sl)] += abs(u) - a[p, d]
                e = [x for x in range(3) if x != d]
                g1, g2 = np.meshgrid(np.arange(n[e[0]]), np.arange(n[e[1]]))
                cells = np.empty((g1.size, 3), np.int32)
                cells[:, e[0]], cells[:, e[1]], cells[:, d] = g1.ravel(), g2.ravel(), face
                nbors = cells.copy()
                nbors[:, d] = n[d] - 1 - face
                links.add(p, cells, [s if x == d else 0 for x in range(3)], q, nbors, u)
        coef.append([diag.ravel()] + [-float(a[p, d]) for d in range(ndim) for _ in (0, 1)])
    box = ((0, 0, 0), (n[0] - 1, n[1] - 1, n[2] - 1))
    if npart == 1 and c["iso"]:  # the plain Laplacian: every entry constant
        coef[0][0] = 2.0 * ndim
    return _system(ndim, P5 if flat else P7, [box] * npart, coef, links)


def _chain(edges, host):
    """Cubes in a row along x, aligned at j = k = 0."""
    a = np.stack([_aniso(host, False) for _ in edges])
    links, coef = _Links(), []
    for p, m in enumerate(edges):
        diag = torch.full((m, m, m), 2.0 * float(a[p].sum()), dtype=torch.float64, device="cuda")
        for s in (-1, 1):
            q = p + s
            if not 0 <= q < len(edges):
                continue
            ov = min(m, edges[q])
            u = -_harm(a[p, 0], a[q, 0])
            face, nface = (m - 1, 0) if s > 0 else (0, edges[q] - 1)
            diag[:ov, :ov, face] += abs(u) - a[p, 0]
            j, k = np.meshgrid(np.arange(ov), np.arange(ov))
            cells = np.stack([np.full(ov * ov, face), j.ravel(), k.ravel()], 1)
            nbors = np.stack([np.full(ov * ov, nface), j.ravel(), k.ravel()], 1)
            links.add(p, cells, [s, 0, 0], q, nbors, u)
        coef.append([diag.ravel()] + [-float(a[p, d]) for d in range(3) for _ in (0, 1)])
    return _system(3, P7, [((0, 0, 0), (m - 1,) * 3) for m in edges], coef, links)


def _stencil_from_kappa(kap, offsets):
    """Harmonic entries to every neighbour inside the box; the diagonal their
    sum plus kappa per missing neighbour."""
    nz, ny, nx = kap.shape
    coef, diag = [None] * len(offsets), torch.zeros_like(kap)
    for e, (ox, oy, oz) in enumerate(offsets[1:], 1):
        off = torch.zeros_like(kap)
        src = tuple(slice(max(0, -o), m - max(0, o)) for o, m in zip((oz, oy, ox), kap.shape))
        dst = tuple(slice(max(0, o), m - max(0, -o)) for o, m in zip((oz, oy, ox), kap.shape))
        off[src] = -_harm(kap[src], kap[dst])
        add = kap.clone()
        add[src] = -off[src]
        diag += add
        coef[e] = off.ravel()
    coef[0] = diag.ravel()
    return coef


def _var27(n, gen):
    nb = -(-n // 8)
    kb = torch.exp(_uniform(nb ** 3, gen, np.log(1e-4), np.log(1e4))).view(nb, nb, nb)
    idx = torch.arange(n, device="cuda") // 8
    kap = kb[idx][:, idx][:, :, idx].contiguous()
    return _system(3, P27, [((0, 0, 0), (n - 1,) * 3)], [_stencil_from_kappa(kap, P27)], _Links())


def _smooth_noise(n, gen):
    g = torch.randn((1, 1, n, n, n), dtype=torch.float64, device="cuda", generator=gen)
    g = torch.nn.functional.avg_pool3d(g, 5, 1, 2, count_include_pad=False)[0, 0]
    return g / g.std()


def _samr(m):
    g0, g1 = m // 4, 3 * m // 4 - 1
    f0, f1 = 2 * g0, 2 * g1 + 1
    cf = 2.0 / 3.0
    ghost = torch.zeros((m, m, m), dtype=torch.bool, device="cuda")
    ghost[g0:g1 + 1, g0:g1 + 1, g0:g1 + 1] = True
    cdiag = torch.zeros((m, m, m), dtype=torch.float64, device="cuda")
    entries = []
    for ox, oy, oz in P7[1:]:
        src = tuple(slice(max(0, -o), m - max(0, o)) for o in (oz, oy, ox))
        dst = tuple(slice(max(0, o), m - max(0, -o)) for o in (oz, oy, ox))
        inb = torch.zeros_like(ghost)
        inb[src] = True
        ng = torch.zeros_like(ghost)
        ng[src] = ghost[dst]
        off = -(inb & ~ghost & ~ng).double()
        cdiag += torch.where(inb, -off, torch.ones_like(off)) + 4 * cf * (inb & ~ghost & ng).double()
        entries.append(off.ravel())
    cdiag[ghost] = 1.0
    fdiag = torch.full((m, m, m), 6.0, dtype=torch.float64, device="cuda")
    for d in range(3):
        for side in (0, m - 1):
            sl = [slice(None)] * 3
            sl[2 - d] = side
            fdiag[tuple(sl)] += cf - 1.0
    links = _Links()
    fa = np.arange(f0, f1 + 1)
    u1, u2 = (v.ravel() for v in np.meshgrid(fa, fa, indexing="ij"))
    for d in range(3):
        for s, fface, cnb in ((-1, f0, g0 - 1), (1, f1, g1 + 1)):
            fc = np.zeros((u1.size, 3), np.int64)
            fc[:, d], fc[:, (d + 1) % 3], fc[:, (d + 2) % 3] = fface, u1, u2
            cc = fc // 2
            cc[:, d] = cnb
            links.add(1, fc, [s if x == d else 0 for x in range(3)], 0, cc, -cf)
            links.add(0, cc, [0, 0, 0], 1, fc, -cf)
    coef = [[cdiag.ravel()] + entries, [fdiag.ravel()] + [-1.0] * 6]
    boxes = [((0, 0, 0), (m - 1,) * 3), ((f0,) * 3, (f1,) * 3)]
    return _system(3, P7, boxes, coef, links), ghost.ravel()


def _batch_edges(c):
    """The problems' shapes are the case's; the seed gives their coefficients."""
    host = np.random.default_rng(c["op"])
    out = []
    for _ in range(c["nprob"]):
        k = int(host.integers(1, 5))
        out.append([int(v) for v in host.integers(c["emin"], c["emax"] + 1, k)])
    return out


def _size(sy):
    return sum(_cells(b) for b in sy["boxes"])


def _cells(box):
    return int(np.prod([h - l + 1 for l, h in zip(*box)]))


def _build(sy):
    grid = S.Grid(sy["ndim"], sy["boxes"])
    A = S.Matrix(grid, sy["offsets"])
    for p, entries in enumerate(sy["coef"]):
        for e, v in enumerate(entries):
            if isinstance(v, float):
                A.set_constant(p, e, v)
            else:
                A.set_box_values(p, e, v)
    if sy["links"] is not None:
        A.add_couplings(*sy["links"])
    A.assemble()
    return A


def _rngs(seed):
    return np.random.default_rng(seed), torch.Generator(device="cuda").manual_seed(seed)


def _describe(c, host, gen):
    """The case's system and, where it has one, the mask of ghost unknowns."""
    if "op" in c:  # the operator is the case's, whatever the seed
        host, gen = _rngs(c["op"])
    if c["kind"] == "grid":
        return _grid(c, host), None
    if c["kind"] == "chain":
        return _chain([int(v) for v in c["edges"].split(",")], host), None
    if c["kind"] == "var27":
        return _var27(c["n"], gen), None
    return _samr(c["m"])


def _rhs(sy, ghost, nrhs, gen):
    b = _uniform((nrhs, _size(sy)), gen)
    if ghost is not None:
        b[:, :ghost.numel()][:, ghost] = 0.0
    return b


def _diffusion(c, gen):
    n = c["n"]
    g = _smooth_noise(n, gen)
    return g, _uniform(n ** 3, gen), _uniform(n ** 3, gen)


# ---------------------------------------------------------------- run ------
def prepare(case, seed):
    host, gen = _rngs(seed)
    do = case["do"]
    if do == "batch":
        systems = [_chain(e, host) for e in _batch_edges(case)]
        B = S.Batch([_build(s) for s in systems], precision=case["precision"],
                    flexible=case["precision"])
        b = _uniform((case["nrhs"], B.num_cells()), gen)
        return {"do": do, "B": B, "b": b, "x": torch.empty_like(b), "nrhs": case["nrhs"]}
    if do == "train":
        g, xt, b = _diffusion(case, gen)
        n = case["n"]
        coef = torch.stack(_stencil_from_kappa(torch.exp(g), P7))
        return {"do": do, "coef": coef.requires_grad_(), "b": b.requires_grad_(), "xt": xt,
                "layout": AD.Layout(3, [((0, 0, 0), (n - 1,) * 3)], P7)}
    if do == "gradient":
        g, lam, x = _diffusion(case, gen)
        n = case["n"]
        sy = _system(3, P7, [((0, 0, 0), (n - 1,) * 3)], [_stencil_from_kappa(torch.exp(g), P7)],
                     _Links())
        sv = S.Solver()
        sv.setup(_build(sy))
        return {"do": do, "sv": sv, "g": g.ravel(), "lam": lam, "x": x, "dg": torch.empty_like(x)}
    sy, ghost = _describe(case, host, gen)
    sv = S.Solver(precision=case["precision"], flexible=case["precision"])
    A = _build(sy)
    if do != "step":
        sv.setup(A)
    b = _rhs(sy, ghost, case.get("nrhs", 1), gen)
    return {"do": do, "A": A, "sv": sv, "b": b, "x": torch.empty_like(b),
            "nrhs": case.get("nrhs", 1)}


def run(state):
    do = state["do"]
    if do == "train":
        x = AD.stencil_solve(state["coef"], state["b"], state["layout"])
        loss = 0.5 * ((x - state["xt"]) ** 2).sum()
        dcoef, db = torch.autograd.grad(loss, (state["coef"], state["b"]))
        return {"x": x.detach(), "dcoef": dcoef, "db": db}
    if do == "gradient":
        state["sv"].diffusion_exp_gradient(state["g"], state["lam"], state["x"], state["dg"])
        return state["dg"]
    if do == "batch":
        state["B"].setup()
        state["B"].solve(state["b"], state["x"], state["nrhs"])
        return state["x"]
    if do == "step":
        state["sv"].setup(state["A"])
    if do in ("step", "solve"):
        state["sv"].solve(state["b"], state["x"], state["nrhs"])
    elif do == "cycle":
        state["sv"].precondition(state["b"], state["x"])
    else:
        state["sv"].level_matvec(0, state["b"], state["x"])
    return state["x"]


# --------------------------------------------------------------- work ------
def work(case):
    """Operator, vectors in and vectors out once; the multiplications and
    additions of one operator apply per right-hand side (solves repeat it a
    number of times that depends on the data)."""
    do, n = case["do"], _unknowns(case)
    if do == "gradient":
        return {"bytes": 32.0 * n, "flops": 60.0 * n}
    if do == "train":
        return {"bytes": 8.0 * n * (7 + 2 + 7 + 2), "flops": 28.0 * n}
    # entries stored per cell (the others are constants), entries per row
    stored = {"var27": 27, "samr": 4}.get(case["kind"], 1)
    per = 27 if case["kind"] == "var27" else 5 if case.get("nz") == 0 else 7
    r = case.get("nrhs", 1)
    return {"bytes": 8.0 * n * (stored + 2 * r), "flops": 2.0 * per * n * r}


# -------------------------------------------------------------- exact ------
class _Plain:
    """The same operator in plain torch: shifted products and an indexed add
    for the couplings."""

    def __init__(self, systems):
        self.parts, rows, cols, vals, diag = [], [], [], [], []
        base = 0
        for sy in systems:
            off = [base]
            for (lo, hi), entries in zip(sy["boxes"], sy["coef"]):
                shape = tuple(hi[d] - lo[d] + 1 for d in (2, 1, 0))
                n = _cells((lo, hi))
                terms = []
                for o, v in zip(sy["offsets"], entries):
                    w = v if isinstance(v, float) else v.view(shape)
                    src = tuple(slice(max(0, -s), m - max(0, s)) for s, m in zip(o[::-1], shape))
                    dst = tuple(slice(max(0, s), m - max(0, -s)) for s, m in zip(o[::-1], shape))
                    if o != (0, 0, 0):
                        terms.append((src, dst, w if isinstance(v, float) else w[src]))
                    else:
                        diag.append(torch.full((n,), v, dtype=torch.float64, device="cuda")
                                    if isinstance(v, float) else v)
                self.parts.append((off[-1], n, shape, terms))
                off.append(off[-1] + n)
            base = off[-1]
            if sy["links"] is not None:
                p, c, _, q, nb, v = sy["links"]
                idx = []
                for part, cell in ((p, c), (q, nb)):
                    lo = np.array([b[0] for b in sy["boxes"]])[part]
                    ext = np.array([np.subtract(b[1], b[0]) + 1 for b in sy["boxes"]])[part]
                    r = cell.astype(np.int64) - lo
                    idx.append(np.array(off)[part] + r[:, 0] + ext[:, 0] * (r[:, 1] + ext[:, 1] * r[:, 2]))
                rows.append(idx[0])
                cols.append(idx[1])
                vals.append(v)
        self.n, self.diag = base, torch.cat(diag)
        self.u = None
        if rows:
            t = [torch.from_numpy(np.concatenate(a)).cuda() for a in (rows, cols, vals)]
            m = torch.sparse_coo_tensor(torch.stack(t[:2]), t[2], (base, base))
            self.u = m.coalesce().to_sparse_csr()

    def __call__(self, x):
        y = self.diag * x
        for o, n, shape, terms in self.parts:
            xv = x[:, o:o + n].view(-1, *shape)
            yv = y[:, o:o + n].view(-1, *shape)
            for src, dst, w in terms:
                yv[(slice(None),) + src] += w * xv[(slice(None),) + dst]
        if self.u is not None:
            y += (self.u @ x.T).T
        return y

    def solve(self, b, limit=12000):
        """CG scaled by the diagonal to 1e-13, checked now and then; None when
        it does not get there."""
        x = torch.zeros_like(b)
        r = b.clone()
        z = r / self.diag
        p = z.clone()
        rz = (r * z).sum(1, keepdim=True)
        stop = 1e-13 * b.norm(dim=1)
        for it in range(limit):
            q = self(p)
            al = rz / (p * q).sum(1, keepdim=True).clamp_min(1e-300)
            x += al * p
            r -= al * q
            z = r / self.diag
            new = (r * z).sum(1, keepdim=True)
            p = z + (new / rz.clamp_min(1e-300)) * p
            rz = new
            if it % 50 == 49 and bool((r.norm(dim=1) <= stop).all()):
                return x
        return None


def exact(case, seed):
    host, gen = _rngs(seed)
    do = case["do"]
    if do == "cycle":
        return None  # a preconditioner's output is not the solution of anything simpler
    if do == "gradient":
        g, lam, x = _diffusion(case, gen)
        n = case["n"]
        kap, lam, x = torch.exp(g), lam.view(n, n, n), x.view(n, n, n)
        acc = torch.zeros_like(kap)
        for d in range(3):
            lo = [slice(None)] * 3
            hi = [slice(None)] * 3
            lo[d], hi[d] = slice(0, n - 1), slice(1, n)
            lo, hi = tuple(lo), tuple(hi)
            s2 = (kap[lo] + kap[hi]) ** 2
            dd = (lam[lo] - lam[hi]) * (x[lo] - x[hi])
            acc[lo] -= 2.0 * kap[hi] ** 2 / s2 * dd
            acc[hi] -= 2.0 * kap[lo] ** 2 / s2 * dd
            for side in (0, n - 1):
                f = [slice(None)] * 3
                f[d] = side
                acc[tuple(f)] -= (lam * x)[tuple(f)]
        return (kap * acc).ravel()
    if do == "train":
        g, xt, b = _diffusion(case, gen)
        n = case["n"]
        sy = _system(3, P7, [((0, 0, 0), (n - 1,) * 3)], [_stencil_from_kappa(torch.exp(g), P7)],
                     _Links())
        A = _Plain([sy])
        x = A.solve(b[None])
        lam = None if x is None else A.solve(x - xt)
        if lam is None:
            return None
        dcoef = torch.zeros((7, n, n, n), dtype=torch.float64, device="cuda")
        xv, lv = x.view(n, n, n), lam.view(n, n, n)
        for e, o in enumerate(P7):
            src = tuple(slice(max(0, -s), n - max(0, s)) for s in o[::-1])
            dst = tuple(slice(max(0, s), n - max(0, -s)) for s in o[::-1])
            dcoef[e][src] = -lv[src] * xv[dst]
        return {"x": x[0], "dcoef": dcoef.view(7, -1), "db": lam[0]}
    if do == "batch":
        systems = [_chain(e, host) for e in _batch_edges(case)]
        A = _Plain(systems)
        b = _uniform((case["nrhs"], A.n), gen)
        return A.solve(b) if b.numel() <= 3 * EXACT_CELLS else None
    sy, ghost = _describe(case, host, gen)
    A = _Plain([sy])
    b = _rhs(sy, ghost, case.get("nrhs", 1), gen)
    if do == "apply":
        return A(b)
    if b.numel() > EXACT_CELLS or case["kind"] == "var27" and case["n"] > 64:
        return None
    return A.solve(b)
