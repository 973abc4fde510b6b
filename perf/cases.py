"""What the solver's speed is measured on: calls of its public entry points as a flow code makes them.

Per time step the projection method solves one pressure Poisson equation (pure Neumann) and one Helmholtz
system per velocity component on an AMR hierarchy; around these it evaluates composite residuals,
interpolates coarse-fine interface data for subcycled levels and, in a differentiable run, solves the
adjoint systems.  Every case below is one such call.  Sizes are those of the repository's workloads and
tests (256^3 + 128^3, 256^2 + 256^2, 96 uneven squares, 4096^2, 64^2, ragged multi-box hierarchies);
``draw`` spreads over the range between them.

Boxes are written as text: levels separated by "|", boxes by ";", "lo:hi" with inclusive indices of the
level, e.g. "192,192,192:319,319,319".
"""
import math

import numpy as np
import torch

from paper_2506_02663_gb300 import amr, autograd

HELMHOLTZ_BETA = -0.25 * 1e-3 / 256.0  # -gamma nu k with gamma = 0.25, nu = 1e-3, k = 1/256
BATCH_SIZES = (64, 96, 128, 192, 256, 384, 512)


# ------------------------------------------------------------------------------------- cases
def listed():
    return [
        # the pressure solve of one 3-D step at the benchmark's size: FP32 V-cycles in FP64 refinement, captured
        {"name": "ppe3d_256", "kind": "solve", "eq": "ppe", "dim": 3, "nx": 256, "ny": 256, "nz": 256,
         "fine": "192,192,192:319,319,319", "precision": "mixed", "graph": True, "cycles": 3},
        # the three velocity components' viscous systems of the same step, in one batched call
        {"name": "helm3d_256", "kind": "components", "dim": 3, "nx": 256, "ny": 256, "nz": 256,
         "fine": "192,192,192:319,319,319", "cycles": 2},
        # a pressure solve on the hierarchy a regridder makes: uneven base, several ragged boxes
        {"name": "ppe3d_boxes", "kind": "solve", "eq": "ppe", "dim": 3, "nx": 96, "ny": 80, "nz": 64,
         "fine": "46,40,32:95,109,81;96,40,32:141,87,81", "precision": "mixed", "graph": True, "cycles": 1},
        # a viscous solve with the default parameters (FP64, host-driven loop)
        {"name": "helm3d_fp64", "kind": "solve", "eq": "helmholtz", "dim": 3, "nx": 72, "ny": 72, "nz": 72,
         "fine": "44,40,36:99,91,107", "precision": "fp64", "graph": False, "cycles": 1},
        # the backward pass of a pressure solve in a differentiable 3-D run
        {"name": "adjoint3d_128", "kind": "adjoint", "eq": "ppe", "dim": 3, "nx": 128, "ny": 128, "nz": 128,
         "fine": "96,96,96:159,159,159", "precision": "mixed"},
        # the smallest solve: single-level Poisson with Dirichlet data, default parameters (launch-bound)
        {"name": "poisson2d_64", "kind": "solve", "eq": "poisson", "dim": 2, "nx": 64, "ny": 64, "nz": 1, "fine": "",
         "precision": "fp64", "graph": False, "cycles": 1},
        # the pressure solve of one two-level 2-D step
        {"name": "ppe2d_256", "kind": "solve", "eq": "ppe", "dim": 2, "nx": 256, "ny": 256, "nz": 1,
         "fine": "128,128:383,383", "precision": "mixed", "graph": True, "cycles": 1},
        # 96 independent uneven 2-D viscous systems (a parameter study) in one call
        {"name": "batch2d_96", "kind": "batch", "dim": 2, "count": 96, "most": 512, "pick": 3},
        # one large uniform 2-D viscous solve
        {"name": "helm2d_4096", "kind": "solve", "eq": "helmholtz", "dim": 2, "nx": 4096, "ny": 4096, "nz": 1, "fine": "",
         "precision": "mixed", "graph": True, "cycles": 1},
        # projection of a velocity and its backward pass on three levels, through autograd (FP64)
        {"name": "project2d_256", "kind": "project", "dim": 2, "nx": 256, "ny": 256, "nz": 1,
         "fine": "102,102:409,409|358,358:665,665"},
        # one composite FP64 residual and its norm: the building block of a user's own iteration
        {"name": "residual3d_256", "kind": "residual", "dim": 3, "nx": 256, "ny": 256, "nz": 256,
         "fine": "192,192,192:319,319,319"},
        # interface data of a subcycled refined level: ghosts at an intermediate time, corrected face averages
        {"name": "cic3d_128", "kind": "cic", "dim": 3, "nx": 256, "ny": 256, "nz": 256,
         "fine": "192,192,192:319,319,319"},
    ]


def _coarsest(n):
    """Cells of the coarsest multigrid grid of a base of ``n`` cells (at most 1024 are accepted)."""
    n = list(n)
    while all(v % 2 == 0 and v >= 8 for v in n):
        n = [v // 2 for v in n]
    return int(np.prod(n))


def _draw_base(rng, dim, low, high):
    """Extents per dimension around a log-uniform size in [low, high], not all equal, accepted by the solver."""
    while True:
        size = math.exp(rng.uniform(math.log(low), math.log(high)))
        n = [max(8, round(size * rng.uniform(0.75, 1.0) / 8) * 8) for _ in range(dim)]
        if rng.random() < 0.3:
            n = [n[0]] * dim
        if max(n) <= high and _coarsest(n) <= 1024:
            return n


def _draw_box(rng, n, lo_frac=0.15, hi_frac=0.5):
    """A box at ratio 2 over cells of a base of extents ``n``, four coarse cells away from the domain faces."""
    lo, hi = [], []
    for v in n:
        w = min(v - 8, max(4, round(v * rng.uniform(lo_frac, hi_frac))))
        a = rng.randint(4, v - 4 - w)
        lo.append(2 * a)
        hi.append(2 * (a + w) - 1)
    return lo, hi


def _box_text(lo, hi):
    return ",".join(map(str, lo)) + ":" + ",".join(map(str, hi))


def _draw_fine(rng, n, pieces):
    """One box, or the box cut in two along its longest extent (boxes that touch)."""
    lo, hi = _draw_box(rng, n)
    if pieces == 1:
        return _box_text(lo, hi)
    d = max(range(len(n)), key=lambda e: hi[e] - lo[e])
    w = (hi[d] - lo[d] + 1) // 2
    cut = lo[d] + 2 * max(2, min(w - 2, round(w * rng.uniform(0.3, 0.7))))
    if hi[d] + 1 - cut < 4 or cut - lo[d] < 4:
        return _box_text(lo, hi)
    h1, l2 = list(hi), list(lo)
    h1[d], l2[d] = cut - 1, cut
    return _box_text(lo, h1) + ";" + _box_text(l2, hi)


def draw(rng):
    kind = rng.choice(("ppe3d", "helm3d", "fp64", "adjoint", "poisson2d", "ppe2d", "batch", "helm2d", "project", "residual", "cic"))
    if kind in ("ppe3d", "helm3d", "fp64", "adjoint"):
        n = _draw_base(rng, 3, 32, 96 if kind == "fp64" else 128 if kind == "adjoint" else 224)
        c = {"dim": 3, "nx": n[0], "ny": n[1], "nz": n[2], "fine": _draw_fine(rng, n, rng.choice((1, 1, 2)))}
        if kind == "ppe3d":
            return {"kind": "solve", "eq": "ppe", "precision": "mixed", "graph": True, "cycles": rng.choice((1, 2, 3)), **c}
        if kind == "helm3d":
            return {"kind": "components", "cycles": rng.choice((1, 2)), **c}
        if kind == "fp64":
            return {"kind": "solve", "eq": "helmholtz", "precision": "fp64", "graph": rng.choice((False, True)), "cycles": 1, **c}
        return {"kind": "adjoint", "eq": rng.choice(("ppe", "helmholtz")), "precision": "mixed", **c}
    if kind == "batch":
        return {"kind": "batch", "dim": 2, "count": rng.randint(3, 96), "most": rng.choice((128, 256, 512)), "pick": rng.randint(0, 999)}
    if kind in ("poisson2d", "ppe2d", "helm2d", "project"):
        n = _draw_base(rng, 2, *{"poisson2d": (16, 256), "ppe2d": (64, 512), "helm2d": (256, 3072), "project": (64, 256)}[kind])
        c = {"dim": 2, "nx": n[0], "ny": n[1], "nz": 1}
        if kind == "poisson2d":
            return {"kind": "solve", "eq": "poisson", "fine": "", "precision": "fp64", "graph": rng.choice((False, True)), "cycles": 1, **c}
        if kind == "helm2d":
            return {"kind": "solve", "eq": "helmholtz", "fine": "", "precision": "mixed", "graph": True, "cycles": 1, **c}
        fine = _draw_fine(rng, n, rng.choice((1, 2)) if kind == "ppe2d" else 1)
        if kind == "ppe2d":
            return {"kind": "solve", "eq": "ppe", "fine": fine, "precision": "mixed", "graph": True, "cycles": 1, **c}
        return {"kind": "project", "fine": fine, **c}
    dim = rng.choice((2, 3))
    n = _draw_base(rng, dim, *((32, 1024) if dim == 2 else (32, 224)))
    return {"kind": kind, "dim": dim, "nx": n[0], "ny": n[1], "nz": n[2] if dim == 3 else 1, "fine": _draw_fine(rng, n, 1)}


# ------------------------------------------------------------------------------------- geometry
def _n0(case):
    return (case["nx"], case["ny"], case["nz"])[:case["dim"]]


def _boxes(case):
    n = _n0(case)
    levels = [[((0,) * len(n), tuple(v - 1 for v in n))]]
    for level in filter(None, case["fine"].split("|")):
        levels.append([tuple(tuple(int(v) for v in end.split(",")) for end in box.split(":")) for box in level.split(";")])
    return levels


def _hierarchy(case):
    return amr.Hierarchy(case["dim"], _n0(case), _boxes(case))


def _batch_sizes(case):
    g = np.random.default_rng(case["pick"])
    n = g.choice([s for s in BATCH_SIZES if s <= case["most"]], size=case["count"])
    nu = np.exp(g.uniform(math.log(1e-4), math.log(1e-2), size=case["count"]))
    return [int(v) for v in n], [-0.25 * float(v) / 256.0 for v in nu]


def _cells(boxes):
    return [sum(int(np.prod([b - a + 1 for a, b in zip(lo, hi)])) for lo, hi in level) for level in boxes]


# ------------------------------------------------------------------------------------- inputs
def _bumps(origin, shape, h, seed, component):
    """Exact cell averages of a sum of eight Gaussian bumps over a block of cells, axes [z,] y, x (double, GPU)."""
    g = np.random.default_rng([seed, component])
    c, w, a = g.uniform(0.0, 1.0, (8, 3)), g.uniform(0.03, 0.1, 8), g.standard_normal(8)
    fac = []
    for d, (o, n) in enumerate(zip(origin, shape)):
        edge = (torch.arange(n + 1, dtype=torch.float64, device="cuda") + o) * h
        t = torch.erf((edge[None, :] - torch.from_numpy(c[:, d:d + 1]).cuda()) / torch.from_numpy(w[:, None]).cuda())
        fac.append((t[:, 1:] - t[:, :-1]) * torch.from_numpy(0.5 * math.sqrt(math.pi) * w[:, None] / h).cuda())
    fac[0] = fac[0] * torch.from_numpy(a[:, None]).cuda()
    return torch.einsum("ax,ay->yx", *fac) if len(fac) == 2 else torch.einsum("ax,ay,az->zyx", *fac)


def _field(hier, seed, component, noise=0.0):
    """A composite field of bumps (plus white noise) on the interior cells, zero in the ghost cells."""
    out = torch.zeros(hier.nelems, dtype=torch.float64, device="cuda")
    for i, p in enumerate(hier.patches):
        block = hier.interior(out, p)
        shape = [b - a + 1 for a, b in zip(p["lo"], p["hi"])]
        block.copy_(_bumps(p["lo"], shape, hier.h0 / 2 ** p["level"], seed, component))
        if noise:
            g = torch.Generator(device="cuda").manual_seed((seed * 1009 + component * 101 + i) % (1 << 31))
            block.add_(torch.randn(block.shape, dtype=torch.float64, device="cuda", generator=g), alpha=noise)
    return out


def _face_data(hier, seed):
    """Smooth Dirichlet face averages: per domain face a cosine of random phase and amplitude."""
    g = np.random.default_rng([seed, 77])
    data = {}
    for f in range(2 * hier.dim):
        n = [hier.n0[e] for e in range(hier.dim) if e != f // 2]
        t = (np.arange(n[0]) + 0.5) / n[0]
        data[f] = g.standard_normal() * np.cos(np.pi * g.integers(1, 4) * t + g.uniform(0, 6.28))
    return data


def _interiors(hier, flat):
    return [hier.interior(flat, p) for p in hier.patches]


def _operator(hier, eq):
    if eq == "helmholtz":
        return amr.Operator(hier, 1.0, HELMHOLTZ_BETA, [amr.DIRICHLET] * (2 * hier.dim))
    return amr.Operator(hier, 0.0, 1.0, [amr.NEUMANN if eq == "ppe" else amr.DIRICHLET] * (2 * hier.dim))


def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind}
    if kind == "batch":
        sizes, betas = _batch_sizes(case)
        s["hiers"] = [amr.Hierarchy(2, (n, n), [[((0, 0), (n - 1, n - 1))]]) for n in sizes]
        s["ops"] = [amr.Operator(h, 1.0, b, [amr.DIRICHLET] * 4) for h, b in zip(s["hiers"], betas)]
        s["fs"] = [_field(h, seed, q) for q, h in enumerate(s["hiers"])]
        s["phis"] = [torch.zeros_like(f) for f in s["fs"]]
        s["params"] = amr.default_params(rtol=1e-10, max_vcycles=100, precision=amr.MIXED, use_graph=1)
        return s
    if kind == "components":  # one hierarchy object per component: their solves run concurrently
        s["hiers"] = [_hierarchy(case) for _ in range(case["dim"])]
        s["ops"] = [_operator(h, "helmholtz") for h in s["hiers"]]
        s["fs"] = [_field(h, seed, q) for q, h in enumerate(s["hiers"])]
        s["phis"] = [torch.zeros_like(f) for f in s["fs"]]
        s["params"] = amr.default_params(rtol=1e-10, max_vcycles=100, precision=amr.MIXED, use_graph=1,
                                         cycles_per_refinement=case["cycles"])
        return s
    h = s["hier"] = _hierarchy(case)
    if kind in ("solve", "adjoint"):
        s["op"] = _operator(h, case["eq"])
        s["f"] = _field(h, seed, 0)
        s["phi"] = torch.zeros_like(s["f"])
        s["bc"] = torch.from_numpy(h.pack_bc([_face_data(h, seed)])).cuda() if case["eq"] == "poisson" else None
        s["params"] = None
        if case["precision"] == "mixed":
            s["params"] = amr.default_params(rtol=1e-10, max_vcycles=100, precision=amr.MIXED,
                                             use_graph=int(kind == "solve" and case["graph"]),
                                             cycles_per_refinement=case.get("cycles", 1))
        elif case["graph"]:
            s["params"] = amr.default_params(use_graph=1)
    elif kind == "project":
        s["op"] = _operator(h, "ppe")
        s["w"] = [_field(h, seed, d, 0.02).requires_grad_() for d in range(case["dim"])]
        s["cot"] = [_field(h, seed, 10 + d, 0.02) for d in range(case["dim"])]
        s["params"] = amr.default_params(rtol=1e-10, max_vcycles=100, use_graph=1)
    elif kind == "residual":
        s["op"] = _operator(h, "helmholtz")
        s["phi"], s["f"] = _field(h, seed, 0, 0.02), _field(h, seed, 1, 0.02)
        s["res"] = torch.zeros_like(s["f"])
    else:  # cic
        s["op"] = _operator(h, "helmholtz")
        s["coarse"] = [[_field(h, seed, 10 * d + t, 0.02) for t in range(4)] for d in range(case["dim"])]
        s["vel"] = [_field(h, seed, 50 + d, 0.02) for d in range(case["dim"])]
        for x in sum(s["coarse"], []) + s["vel"]:
            s["op"].fill_ghosts(x)
        s["rate"] = [torch.zeros_like(x) for x in s["vel"]]
        info = amr.cic_faces(h, 1)
        s["faces"] = torch.zeros(len(info["face"]), dtype=torch.float64, device="cuda")
        s["delta"] = torch.zeros(info["ncomponents"], dtype=torch.float64, device="cuda")
    return s


# ------------------------------------------------------------------------------------- the calls
def run(s):
    kind = s["kind"]
    if kind in ("batch", "components"):
        amr.batch_solve(s["ops"], s["phis"], s["fs"], params=s["params"])
        if kind == "components":
            return [_interiors(h, x) for h, x in zip(s["hiers"], s["phis"])]
        return torch.cat(s["phis"])  # problem after problem in one array (the ghost cells stay zero)
    h = s["hier"]
    if kind == "solve":
        s["op"].solve(s["phi"], s["f"], bc=s["bc"], params=s["params"])
        return _interiors(h, s["phi"])
    if kind == "adjoint":
        s["op"].solve_transpose(s["phi"], s["f"], params=s["params"])
        return _interiors(h, s["phi"])
    if kind == "project":
        u = autograd.project(s["op"], [amr.DIRICHLET] * (2 * h.dim), s["w"], s["params"])
        grads = torch.autograd.grad(u, s["w"], s["cot"])
        return {"u": [_interiors(h, x) for x in u], "grad": [_interiors(h, x) for x in grads]}
    if kind == "residual":
        norm = s["op"].residual(s["phi"], s["f"], s["res"])
        return {"res": _interiors(h, s["res"]), "norm": norm}
    k = h.h0
    for d in range(h.dim):
        amr.cic_ghosts(h, 1, s["coarse"][d], k, 0.5 * k, s["vel"][d], s["rate"][d])
    amr.cic_face_averages(h, 1, s["vel"], s["faces"], delta=s["delta"])
    at = h.patches[1]["offset"]
    return {"value": [x[at:] for x in s["vel"]], "rate": [x[at:] for x in s["rate"]], "faces": s["faces"], "delta": s["delta"]}


def work(case):
    """Each input field read once and each output field written once, 8 bytes a value; operations of one
    application of the operator per unknown (a solve needs at least one of them)."""
    if case["kind"] == "batch":
        cells = sum(n * n for n in _batch_sizes(case)[0])
        return {"bytes": 16 * cells, "flops": 12 * cells}
    D, cells = case["dim"], _cells(_boxes(case))
    total = sum(cells)
    apply = (6 * D + 2) * total
    if case["kind"] in ("solve", "adjoint"):
        return {"bytes": 16 * total, "flops": apply}
    if case["kind"] == "components":
        return {"bytes": 16 * D * total, "flops": D * apply}
    if case["kind"] == "project":  # w, u, the incoming and the outgoing gradients
        return {"bytes": 32 * D * total, "flops": 4 * apply}
    if case["kind"] == "residual":
        return {"bytes": 24 * total, "flops": apply}
    lo, hi = _boxes(case)[1][0]
    n = [b - a + 1 for a, b in zip(lo, hi)]
    area = [int(np.prod(n)) // v for v in n]
    ghosts = sum(4 * a for a in area)  # two layers on two sides
    # coarse window cells: the ghosts' parents (one layer per side), two more on both sides of it
    window = sum(2 * 5 * int(np.prod([n[e] // 2 + 4 for e in range(D) if e != d])) for d in range(D))
    return {"bytes": 8 * D * (4 * window + 2 * ghosts) + 40 * sum(2 * a for a in area),
            "flops": 2 * D * (8 * window + 2 * (2 * 5 ** D + 4 * 5 ** (D - 1) + 8 * 5 ** (D - 2)) * ghosts // 2 ** D)}


# ------------------------------------------------------------------------------------- 64-bit references
# Ghost values from the four cells next to a face, layer 1 and 2: homogeneous part and data coefficient.
_GHOST = {0: (np.array([[-77, 43, -17, 3], [-505, 335, -145, 27]]) / 12.0, np.array([5.0, 25.0])),
          1: (np.array([[5, 9, -5, 1], [-75, 145, -75, 15]]) / 10.0, np.array([6.0 / 5.0, 6.0]))}


def _line_matrix(n, h, bc):
    """The 1-D fourth-order second derivative on n cells with homogeneous ghosts of type ``bc`` at both ends
    and the coefficients of the face data of the low end (of the high end: reversed)."""
    ext = np.zeros((n + 4, n))
    ext[2:n + 2] = np.eye(n)
    for layer in (0, 1):
        ext[1 - layer, :4] = _GHOST[bc][0][layer]
        ext[n + 2 + layer, n - 4:] = _GHOST[bc][0][layer][::-1]
    data = np.zeros(n + 4)
    data[1], data[0] = _GHOST[bc][1]
    st = lambda m: (-m[:-4] + 16 * m[1:-3] - 30 * m[2:-2] + 16 * m[3:-1] - m[4:]) / (12 * h * h)  # noqa: E731
    return st(ext), st(data)


def _solve_single(f, h, alpha, beta, bc, faces=None):
    """(alpha + beta L) phi = f on one uniform 2-D grid, f[y, x]: the separable operator diagonalised per direction."""
    f = f.copy()
    ny, nx = f.shape
    (mx, dx), (my, dy) = _line_matrix(nx, h, bc), _line_matrix(ny, h, bc)
    if faces is not None:
        f -= beta * (np.outer(faces[0], dx) + np.outer(faces[1], dx[::-1]) + np.outer(dy, faces[2]) + np.outer(dy[::-1], faces[3]))
    lx, vx = np.linalg.eig(mx)
    ly, vy = (lx, vx) if nx == ny else np.linalg.eig(my)
    t = np.linalg.solve(vy, f) @ np.linalg.inv(vx).T
    t = t / (alpha + beta * (ly[:, None] + lx[None, :]))
    return np.ascontiguousarray((vy @ t @ vx.T).real)


def _cfi_matrix(n):
    """Conservative quartic interpolation of n coarse cell averages to the 2 (n - 4) fine ones of the inner cells."""
    edges = np.arange(-2.5, 3.0)
    rows = []
    for a, b in ((-0.5, 0.0), (0.0, 0.5)):
        basis = lambda x: np.array([np.prod([(x - edges[k]) / (edges[j] - edges[k]) for k in range(6) if k != j]) for j in range(6)])  # noqa: E731
        v = (basis(b) - basis(a)) / (b - a)  # average of the primitive's derivative over the fine cell
        rows.append([v[j + 1:].sum() for j in range(5)])  # primitive values are running sums of the averages
    out = np.zeros((2 * (n - 4), n))
    for i in range(n - 4):
        out[2 * i, i:i + 5], out[2 * i + 1, i:i + 5] = rows
    return torch.from_numpy(out).cuda()


def _cut(x, d, a, b):
    """Slice [a, b) of dimension d of an array with axes [z,] y, x."""
    return x.narrow(x.dim() - 1 - d, a, b - a)


def _interpolated(coarse, lo, hi):
    """AMRCFI of a coarse level over the box [lo, hi] of the next level grown by two cells."""
    x = coarse
    for d, (a, b) in enumerate(zip(lo, hi)):
        x = _cut(x, d, a // 2 - 3, (b + 1) // 2 + 3)
    for d in range(len(lo)):
        axis = x.dim() - 1 - d
        x = torch.movedim(torch.tensordot(_cfi_matrix(x.shape[axis]), x, dims=([1], [axis])), 0, axis)
    return x


def _averaged(fine):
    for d in range(fine.dim()):
        n = fine.shape[fine.dim() - 1 - d]
        fine = 0.5 * (fine.unflatten(fine.dim() - 1 - d, (n // 2, 2)).sum(fine.dim() - d))
    return fine


def _covered(x, lo, hi):
    for d, (a, b) in enumerate(zip(lo, hi)):
        x = _cut(x, d, a // 2, (b + 1) // 2)
    return x


def _second(ext, d, n):
    """12 h^2 times the second derivative along d of an array extended by two cells there."""
    return 16 * (_cut(ext, d, 1, n + 1) + _cut(ext, d, 3, n + 3)) - _cut(ext, d, 0, n) - _cut(ext, d, 4, n + 4) - 30 * _cut(ext, d, 2, n + 2)


def _exact_residual(case, seed):
    s = prepare(case, seed)
    h, D = s["hier"], case["dim"]
    (pc, pf), (lo, hi) = h.patches, _boxes(case)[1][0]
    c, f = h.interior(s["phi"], pc).clone(), h.interior(s["phi"], pf)
    _covered(c, lo, hi).copy_(_averaged(f))
    big = _interpolated(c, lo, hi)
    hc, hf = h.h0, h.h0 / 2
    lc, lf = torch.zeros_like(c), torch.zeros_like(f)
    g0 = _GHOST[0][0]
    for d in range(D):
        n, m = c.shape[D - 1 - d], f.shape[D - 1 - d]
        low = [sum(g0[layer][q] * _cut(c, d, q, q + 1) for q in range(4)) for layer in (0, 1)]
        high = [sum(g0[layer][q] * _cut(c, d, n - 1 - q, n - q) for q in range(4)) for layer in (0, 1)]
        lc += _second(torch.cat([low[1], low[0], c, high[0], high[1]], D - 1 - d), d, n) / (12 * hc * hc)
        strip = big
        for e in range(D):
            if e != d:
                strip = _cut(strip, e, 2, 2 + f.shape[D - 1 - e])
        ext = torch.cat([_cut(strip, d, 0, 2), f, _cut(strip, d, m + 2, m + 4)], D - 1 - d)
        lf += _second(ext, d, m) / (12 * hf * hf)
        flux = lambda x, a, hx: (_cut(x, d, a, a + 1) - 15 * _cut(x, d, a + 1, a + 2) + 15 * _cut(x, d, a + 2, a + 3) - _cut(x, d, a + 3, a + 4)) / (12 * hx)  # noqa: E731
        for side in (0, 1):  # the coarse cell outside the box: its flux replaced by the mean of the fine fluxes
            at = lo[d] // 2 if side == 0 else (hi[d] + 1) // 2  # the coarse face's upper cell
            cl, fl = c, flux(ext, 0 if side == 0 else m, hf)
            for e in range(D):
                if e != d:
                    cl = _cut(cl, e, lo[e] // 2, (hi[e] + 1) // 2)
                    ax = D - 1 - e
                    fl = 0.5 * fl.unflatten(ax, (fl.shape[ax] // 2, 2)).sum(ax + 1)
            corr = (fl - flux(cl, at - 2, hc)) / hc
            cell = _cut(lc, d, at - 1, at) if side == 0 else _cut(lc, d, at, at + 1)
            for e in range(D):
                if e != d:
                    cell = _cut(cell, e, lo[e] // 2, (hi[e] + 1) // 2)
            cell += corr if side == 0 else -corr
    rc = h.interior(s["f"], pc) - (c + HELMHOLTZ_BETA * lc)
    rf = h.interior(s["f"], pf) - (f + HELMHOLTZ_BETA * lf)
    _covered(rc, lo, hi).zero_()
    norm = max(float(rc.abs().max()), float(rf.abs().max()))
    _covered(rc, lo, hi).copy_(_averaged(rf))
    return {"res": [rc, rf], "norm": norm}


def _exact_cic(case, seed):
    s = prepare(case, seed)
    h, D = s["hier"], case["dim"]
    (pc, pf), (lo, hi) = h.patches, _boxes(case)[1][0]
    k = h.h0
    # cubic Lagrange weights (and slopes) at t* = t_{-1} + k/2 of the times t_{-3}, .., t_{-0} at -2k, -k, 0, k
    t, x = np.array([1.0, 0.0, -1.0, -2.0]) * k, 0.5 * k  # of coarse[0], .., coarse[3]
    w = [[], []]
    for i in range(4):
        o = [t[q] for q in range(4) if q != i]
        den = np.prod([t[i] - v for v in o])
        w[0].append(np.prod([x - v for v in o]) / den)
        w[1].append(((x - o[1]) * (x - o[2]) + (x - o[0]) * (x - o[2]) + (x - o[0]) * (x - o[1])) / den)
    out = {"value": [], "rate": [], "faces": None, "delta": None}
    at = pf["offset"]
    for d in range(D):
        for name, weights, base in (("value", w[0], s["vel"][d]), ("rate", w[1], s["rate"][d])):
            big = _interpolated(sum(weights[q] * h.interior(s["coarse"][d][q], pc) for q in range(4)), lo, hi)
            flat = base.clone()
            patch = h._view(flat, pf)
            for e in range(D):
                n = [b - a + 1 for a, b in zip(lo, hi)]
                for a, b in ((0, 2), (n[e] + 2, n[e] + 4)):
                    dst, src = patch, big
                    for q in range(D):
                        r = (a, b) if q == e else (2, 2 + n[q])
                        dst, src = _cut(dst, q, *r), _cut(src, q, *r)
                    dst.copy_(src)
            out[name].append(flat[at:])
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "residual":
        return _exact_residual(case, seed)
    if kind == "cic":
        return _exact_cic(case, seed)
    if kind == "batch":
        sizes, betas = _batch_sizes(case)
        out = []
        for q, (n, b) in enumerate(zip(sizes, betas)):
            phi = _solve_single(_bumps((0, 0), (n, n), 1.0 / n, seed, q).cpu().numpy(), 1.0 / n, 1.0, b, 0)
            out.append(amr.Hierarchy(2, (n, n), [[((0, 0), (n - 1, n - 1))]]).pack([[phi.T]]))
        return np.concatenate(out)
    if kind == "solve" and case["dim"] == 2 and not case["fine"] and max(_n0(case)) <= 512:
        nx, ny = _n0(case)
        f = _bumps((0, 0), (nx, ny), 1.0 / nx, seed, 0).cpu().numpy()
        if case["eq"] == "poisson":
            faces = _face_data(amr.Hierarchy(2, (nx, ny), _boxes(case)), seed)
            return [_solve_single(f, 1.0 / nx, 0.0, 1.0, 0, faces)]
        return [_solve_single(f, 1.0 / nx, 1.0, HELMHOLTZ_BETA, 0)]
    return None  # composite solves: no direct solution in a few seconds
