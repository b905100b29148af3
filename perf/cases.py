"""Performance cases of the framework: the calls a room-acoustics program makes, over the sizes it makes them at.

A case is a dict of plain values: what is called (``kind``), the room and its mesh, the frequency, and the options
of the operator.  ``prepare`` builds what such a program keeps (mesh, octree, operators with their saved translation
forms, preconditioners, input vectors), ``run`` makes one pass through the public entry points, ``work`` counts the
bytes and operations a pass cannot do without, and ``exact`` computes the same result as a dense sum in 64 bits.

Kinds:
  matvec   one FMM matrix-vector product, the step every Krylov iteration makes
  multi    the same for several right-hand sides at once (all sources of one frequency)
  solve    one FGMRES solve with the inner-outer preconditioner, judged by the FP64 operator
  sweep    fb_batch_solve over a few frequencies: operator construction and solves
  field    the field at receivers from a boundary solution
  setup    construction of a mixed operator and its block Jacobi, then one product with each
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2103_16073_gb300 as fb
from paper_2103_16073_gb300 import workloads as W

SOUND_SPEED = W.SOUND_SPEED
LEAF_MAX = 64
RESTART = 40
TOL = 1e-4
INNER_STEPS = 14                   # inner GMRES steps and order rule of the inner-outer preconditioner
INNER_D0, INNER_PMIN = 0.5, 2
SHOEBOX = (3.0, 2.4, 2.0)          # m


def _shoebox(kind, name, counts, freq, room=SHOEBOX, **more):
    c = {"kind": kind, "room": "shoebox", "lx": room[0], "ly": room[1], "lz": room[2],
         "nx": counts[0], "ny": counts[1], "nz": counts[2], "freq": freq}
    if name:
        c["name"] = name
    return {**c, **more}


def _lroom(kind, name, freq, per_wavelength=8.0, **more):
    c = {"kind": kind, "room": "lroom", "freq": freq, "per_wavelength": per_wavelength}
    if name:
        c["name"] = name
    return {**c, **more}


MIXED = {"precision": "mixed", "d0": 6.0, "pmin": 12}
FP64 = {"precision": "fp64", "d0": 6.0, "pmin": 12}
INNER = {"precision": "mixed16", "d0": INNER_D0, "pmin": INNER_PMIN}   # mixed with BF16 near-field entries


def listed():
    return [
        # the smallest product of a sweep: a low frequency on 3,072 elements, a chain of short launches
        _shoebox("matvec", "matvec_small_125hz", (16, 16, 16), 125.0, **MIXED),
        # the ordinary product: the shoebox room at 1 kHz, 39,368 elements at lambda/8
        _shoebox("matvec", "matvec_shoebox_1khz", (70, 56, 47), 1000.0, **MIXED),
        # the top of a broadband sweep: the L-shaped room at 2 kHz, 567,592 elements, orders 12 to 88
        _lroom("matvec", "matvec_lroom_2khz", 2000.0, **MIXED),
        # large expansion orders (116 and 66): a mesh that is coarse for its frequency
        _shoebox("matvec", "matvec_high_order", (16, 16, 16), 7500.0, **MIXED),
        # the low-accuracy product that the inner-outer preconditioner makes many of per outer iteration
        _lroom("matvec", "inner_lroom_2khz", 2000.0, **INNER),
        # the FP64 product that judges the true residual, at the ordinary and at the largest size
        _shoebox("matvec", "judge_shoebox_1khz", (70, 56, 47), 1000.0, **FP64),
        _lroom("matvec", "judge_lroom_2khz", 2000.0, **FP64),
        # all eight sources of one frequency of the sweep in lockstep
        _lroom("multi", "sources_lroom_600hz", 609.2, nrhs=8, **MIXED),
        # one whole solve at 1e-4: FGMRES, inner-outer preconditioner, FP64 true residual
        _shoebox("solve", "solve_shoebox_1khz", (70, 56, 47), 1000.0, **MIXED),
        # the low end of a frequency sweep through the batch scheduler, operators built on the way
        _lroom("sweep", "sweep_lroom_low", 100.0, freq_hi=200.0, jobs=3, nsrc=8, inner=INNER_STEPS, **MIXED),
        # the field at 1,024 receivers from the solution on the shoebox room
        _shoebox("field", "receivers_shoebox_1khz", (70, 56, 47), 1000.0, nrec=1024, **FP64),
        # what every new frequency pays before its first product
        _lroom("setup", "setup_lroom_600hz", 609.2, **MIXED),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _draw_shoebox(rng, n, per_wavelength):
    """A room of about the shoebox's proportions meshed with about n elements; its frequency makes the legs
    lambda / per_wavelength."""
    lx, ly, lz = (round(rng.uniform(a, b), 3) for a, b in ((2.0, 6.5), (1.8, 5.5), (1.6, 4.2)))
    h = math.sqrt(4.0 * (lx * ly + lx * lz + ly * lz) / n)
    counts = [max(3, int(round(v / h))) for v in (lx, ly, lz)]
    leg = max(lx / counts[0], ly / counts[1], lz / counts[2])
    return (lx, ly, lz), counts, round(SOUND_SPEED / (per_wavelength * leg), 2)


def draw(rng):
    kind = rng.choice(["mixed", "mixed", "mixed", "inner", "fp64", "coarse", "multi", "solve", "sweep", "field", "setup"])
    if kind == "sweep":
        lo = round(_log(rng, 80.0, 130.0), 2)
        return _lroom("sweep", "", lo, freq_hi=round(lo * rng.uniform(1.2, 1.5), 2), jobs=rng.randint(1, 3),
                      nsrc=rng.randint(1, 8), inner=rng.choice([0, INNER_STEPS]), **MIXED)
    if kind == "coarse":   # high orders: element legs near or above one wavelength
        room, counts, f = _draw_shoebox(rng, _log(rng, 1500, 4000), rng.uniform(0.4, 1.0))
        f = min(f, 7500.0 * 3.0 / max(room))   # no larger electrically than the listed one
        return _shoebox("matvec", "", counts, round(f, 2), room, **MIXED)
    opts = {"inner": INNER, "fp64": FP64, "field": FP64}.get(kind, MIXED)
    # smallest and largest element counts of the kind, spread over their logarithm
    lo, hi = {"mixed": (1200, 560000), "inner": (1200, 560000), "fp64": (1200, 300000), "multi": (1200, 60000),
              "solve": (1200, 60000), "field": (1200, 60000), "setup": (1200, 100000)}[kind]
    n = _log(rng, lo, hi)
    more = {}
    if kind == "multi":
        more["nrhs"] = rng.choice([2, 3, 4, 5, 8])
    if kind == "field":
        more["nrec"] = int(_log(rng, 16, 1024))
    call = {"mixed": "matvec", "inner": "matvec", "fp64": "matvec"}.get(kind, kind)
    if n > 4000 and rng.random() < 0.35:   # the L-shaped room: 142 m^2 of walls, two triangles per rectangle
        h = math.sqrt(2.0 * 142.0 / n)
        ppw = rng.uniform(6.0, 10.0)
        return _lroom(call, "", round(SOUND_SPEED / (ppw * h), 2), round(ppw, 2), **more, **opts)
    room, counts, f = _draw_shoebox(rng, n, rng.uniform(6.0, 12.0))
    return _shoebox(call, "", counts, f, room, **more, **opts)


# ------------------------------------------------------------------ state ----
def _mesh_of(case, freq=None):
    """(verts, tris, wall index) of a case, at another frequency of a sweep if given."""
    if case["room"] == "lroom":
        return W.lroom_mesh(SOUND_SPEED / (freq or case["freq"]) / case["per_wavelength"])
    return W.shoebox_mesh(case["lx"], case["ly"], case["lz"], case["nx"], case["ny"], case["nz"])


def _interior_points(case, rng, n, margin):
    """Points of the room at least `margin` from its bounding walls."""
    if case["room"] == "lroom":
        out = []
        while len(out) < n:
            p = np.array([8.0, 4.0, 3.0]) * rng.random(3)
            if W.lroom_inside(p, margin)[0]:
                out.append(p)
        return np.asarray(out)
    return W.uniform_points_in_box(rng, [0, 0, 0], [case["lx"], case["ly"], case["lz"]], n, margin)


def _inputs(case, seed):
    """What the seed decides: one admittance per wall and the points of sources and receivers."""
    rng = np.random.Generator(np.random.PCG64(int(seed)))
    beta_wall = rng.uniform(0.05, 0.5, size=10)
    src = _interior_points(case, rng, max(1, int(case.get("nsrc", 1))), 0.3)
    rec = _interior_points(case, rng, int(case.get("nrec", 0)), 0.3) if case.get("nrec") else None
    return beta_wall, src, rec


def _rough_vectors(seed, n, rows):
    """Krylov-like vectors: oscillating along the walls and rough, of unit size."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    return torch.randn((rows, n), dtype=torch.complex128, device="cuda", generator=g)


class _State:
    """The handles of one prepared case; they are released with it."""

    def __init__(self, case):
        self.case = case
        self._handles = []

    def keep(self, handle, destroy):
        self._handles.append((handle, destroy))
        return handle

    def __del__(self):
        while self._handles:
            handle, destroy = self._handles.pop()
            destroy(handle)


def _geometry(s, case, beta_wall, freq=None):
    verts, tris, wall = _mesh_of(case, freq)
    mesh = s.keep(fb.fb_mesh_create(verts, tris), fb.fb_mesh_destroy)
    fb.fb_mesh_set_admittance(mesh, beta_wall[wall].astype(np.complex128))
    tree = s.keep(fb.fb_tree_build(mesh, LEAF_MAX), fb.fb_tree_destroy)
    return mesh, tree, tris.shape[0]


def _saved_forms(op, tree, fp64):
    """Translation forms per level as a program restores them from an earlier autotuned run on this card: staged
    passes for large orders (on the tensor cores in mixed precision, in double-FP32 in FP64), composed tensor-core
    matrices for small orders on levels of many boxes, per-pair tiles for the rest."""
    boxes = fb.fb_tree_info(tree)[3]
    _, top, p = fb.fb_operator_info(op)
    forms = [0] * 13
    for lev in range(2, top + 1):
        pair = max(int(p[lev]), int(p[lev - 1])) if lev > 2 else 0
        if fp64:
            forms[lev] = 4 + 64 if p[lev] >= 60 else 256
            if pair:
                forms[lev] |= 8 + 128 if pair >= 60 else 512
        else:
            if p[lev] >= 26:
                forms[lev] = 4 + 16 + 1024
            elif p[lev] <= 20 and (boxes[lev] >= 1000 or p[lev] <= 8):
                forms[lev] = 1
            if pair >= 100:
                forms[lev] |= 8 + 32 + 2048
            elif pair >= 24:
                forms[lev] |= 8
            elif pair and pair <= 8 and boxes[lev] >= 20000:
                forms[lev] |= 2
    return forms


def _operator(s, case, mesh, tree, kind, precision, d0, pmin, tuned=True, donor=None):
    code = fb.FB_PREC_FP64_FMM if precision == "fp64" else fb.FB_PREC_MIXED_FMM
    if donor is not None:
        op = fb.fb_operator_create_like(donor, code, d0, pmin)
    else:
        op = fb.fb_operator_create(mesh, tree, W.wavenumber(case["freq"]), kind, code, d0, pmin)
    s.keep(op, fb.fb_operator_destroy)
    if tuned:
        fb.fb_operator_set_forms(op, _saved_forms(op, tree, precision == "fp64"))
    if precision == "mixed16":
        fb.fb_operator_set_near_bf16(op, True)
    return op


def prepare(case, seed):
    s = _State(case)
    beta_wall, src, rec = _inputs(case, seed)
    kind = case["kind"]
    k = W.wavenumber(case["freq"])
    if kind == "sweep":
        s.jobs = []
        for f in np.geomspace(case["freq"], case["freq_hi"], int(case["jobs"])):
            mesh, tree, n = _geometry(s, case, beta_wall, f)
            x = torch.zeros((src.shape[0], n), dtype=torch.complex128, device="cuda")
            s.jobs.append({"mesh": mesh, "tree": tree, "k": W.wavenumber(f), "src": src, "x": x})
        return s
    s.mesh, s.tree, s.n = _geometry(s, case, beta_wall)
    if kind == "field":
        s.k, s.src = k, src[0]
        s.gamma = torch.empty(s.n, dtype=torch.complex128, device="cuda")
        fb.fb_gamma_monopole(s.mesh, k, s.src, s.gamma)
        s.psi = torch.empty_like(s.gamma)   # a wave field on the walls, as a solution is
        fb.fb_gamma_monopole(s.mesh, k, src[0] + np.array([0.05, -0.04, 0.03]), s.psi)
        s.psi /= k
        s.rec = torch.tensor(rec, device="cuda")
        s.out = torch.empty(rec.shape[0], dtype=torch.complex128, device="cuda")
        return s
    if kind == "solve":
        judge = _operator(s, case, s.mesh, s.tree, fb.FB_OP_A, "fp64", case["d0"], case["pmin"])
        s.op = _operator(s, case, s.mesh, s.tree, fb.FB_OP_A, "mixed", case["d0"], case["pmin"], donor=judge)
        single = _operator(s, case, s.mesh, s.tree, fb.FB_OP_L, "fp64", case["d0"], case["pmin"])
        low = _operator(s, case, s.mesh, s.tree, fb.FB_OP_A, "mixed16", INNER_D0, INNER_PMIN, donor=judge)
        jacobi = s.keep(fb.fb_precond_create(low, fb.FB_PC_BLOCK_JACOBI), fb.fb_precond_destroy)
        for op in (s.op, judge, low):
            fb.fb_operator_use_graphs(op, True)
        s.pc = s.keep(fb.fb_precond_create_inner(s.op, low, jacobi, INNER_STEPS), fb.fb_precond_destroy)
        fb.fb_precond_use_graphs(s.pc, True)
        s.judge = judge
        gamma = torch.empty(s.n, dtype=torch.complex128, device="cuda")
        fb.fb_gamma_monopole(s.mesh, k, src[0], gamma)
        s.b = torch.empty_like(gamma)
        fb.fb_operator_apply(single, gamma, s.b)
        s.x = torch.zeros_like(s.b)
        return s
    rows = int(case.get("nrhs", 1))
    s.x = _rough_vectors(seed, s.n, rows)
    gamma = torch.empty(s.n, dtype=torch.complex128, device="cuda")
    fb.fb_gamma_monopole(s.mesh, k, src[0], gamma)
    s.x += gamma * (math.sqrt(s.n) / torch.linalg.vector_norm(gamma))
    s.y = torch.empty_like(s.x)
    if kind != "setup":
        s.op = _operator(s, case, s.mesh, s.tree, fb.FB_OP_A, case["precision"], case["d0"], case["pmin"])
    if kind != "multi":
        s.x, s.y = s.x[0], s.y[0]
    if kind == "setup":
        s.k, s.z = k, torch.empty_like(s.y)
    return s


def run(state):
    s = state
    kind = s.case["kind"]
    if kind == "matvec":
        return fb.fb_operator_apply(s.op, s.x, s.y)
    if kind == "multi":
        return fb.fb_operator_apply_multi(s.op, s.x, s.y)
    if kind == "solve":
        s.x.zero_()
        fb.fb_fgmres_solve(s.op, s.b, s.x, pc=s.pc, tol=TOL, restart=RESTART, true_op=s.judge)
        return s.x
    if kind == "sweep":
        for job in s.jobs:
            job["x"].zero_()
        fb.fb_batch_solve(s.jobs, tol=TOL, restart=RESTART, autotune=False, max_rhs=8,
                          inner_iters=int(s.case["inner"]))
        return [job["x"] for job in s.jobs]
    if kind == "field":
        return fb.fb_eval_field(s.mesh, s.k, s.psi, s.gamma, s.rec, s.out, src=s.src)
    # setup
    c = s.case
    op = fb.fb_operator_create(s.mesh, s.tree, s.k, fb.FB_OP_A, fb.FB_PREC_MIXED_FMM, c["d0"], c["pmin"])
    pc = fb.fb_precond_create(op, fb.FB_PC_BLOCK_JACOBI)
    fb.fb_operator_apply(op, s.x, s.y)
    fb.fb_precond_apply(pc, s.x, s.z)
    fb.fb_precond_destroy(pc)
    fb.fb_operator_destroy(op)
    return [s.y, s.z]


# ------------------------------------------------------------------- work ----
def _order(k, side, d0, pmin):
    kr = k * math.sqrt(3.0) / 2.0 * side
    return max(int(pmin), math.ceil(kr + 1.8 * d0 ** (2.0 / 3.0) * kr ** (1.0 / 3.0)))


def _product_work(case, freq, precision, d0, pmin):
    """(bytes, flops, elements, near entries) of one FMM product: every near-field entry and P2M / L2P row read
    once, the vectors read and written once; 8 flops per near-field, P2M and L2P entry, and per box pair two folded
    rotations (4 flops per real x complex entry) and the coaxial blocks (8 per entry)."""
    s = _State(case)
    mesh, tree, n = _geometry(s, case, np.full(10, 0.2), freq)
    top, _, side, boxes = fb.fb_tree_info(tree)
    k = W.wavenumber(freq)
    start = fb.fb_tree_export(tree, 1)
    occ = np.diff(start)
    u = fb.fb_tree_export(tree, 3)
    near = float(np.sum(occ[u[:, 0]] * occ[u[:, 1]]))
    p = [_order(k, side / 2 ** lev, d0, pmin) if lev >= 2 else 0 for lev in range(top + 1)]

    def rot(q):
        return 4.0 * sum((j + 1) ** 2 + j ** 2 for j in range(q))

    def pair(a, b):
        q = min(a, b)
        return rot(a) + rot(b) + 8.0 * sum((a - abs(m)) * (b - abs(m)) for m in range(-q + 1, q))

    flops = 8.0 * near + 16.0 * n * p[top] ** 2
    for lev in range(2, top + 1):
        flops += fb.fb_tree_export(tree, 4, lev).shape[0] * pair(p[lev], p[lev])
        if lev > 2:
            flops += 2.0 * float(boxes[lev]) * pair(p[lev], p[lev - 1])
    size = 16 if precision == "fp64" else 8
    entry = 4 if precision == "mixed16" else size
    return near * entry + 2.0 * n * p[top] ** 2 * size + 32.0 * n, flops, n, near


def work(case):
    kind = case["kind"]
    if kind in ("matvec", "multi"):
        b, f, n, _ = _product_work(case, case["freq"], case["precision"], case["d0"], case["pmin"])
        r = int(case.get("nrhs", 1))
        return {"bytes": b + 32.0 * n * (r - 1), "flops": f * r}
    if kind == "field":
        n = 4 * (case["nx"] * case["ny"] + case["nx"] * case["nz"] + case["ny"] * case["nz"]) \
            if case["room"] == "shoebox" else _mesh_of(case)[1].shape[0]
        # 3 Gauss points per element and receiver, about 40 operations each
        return {"bytes": n * (9 + 3 + 1 + 2 + 4) * 8.0 + case["nrec"] * 40.0, "flops": 120.0 * n * case["nrec"]}
    if kind == "setup":
        b, f, n, near = _product_work(case, case["freq"], "mixed", case["d0"], case["pmin"])
        return {"bytes": 2.0 * b, "flops": f + 120.0 * near}
    if kind == "solve":   # four outer iterations are usual: a mixed product, 14 inner ones each; one FP64 product
        b, f, n, _ = _product_work(case, case["freq"], "mixed", case["d0"], case["pmin"])
        bi, fi, _, _ = _product_work(case, case["freq"], "mixed16", INNER_D0, INNER_PMIN)
        bj, fj, _, _ = _product_work(case, case["freq"], "fp64", case["d0"], case["pmin"])
        return {"bytes": 4 * b + 4 * INNER_STEPS * bi + bj, "flops": 4 * f + 4 * INNER_STEPS * fi + fj}
    total = {"bytes": 0.0, "flops": 0.0}
    r = int(case["nsrc"])
    for freq in np.geomspace(case["freq"], case["freq_hi"], int(case["jobs"])):
        b, f, n, near = _product_work(case, freq, "mixed", case["d0"], case["pmin"])
        bj, fj, _, _ = _product_work(case, freq, "fp64", case["d0"], case["pmin"])
        # the near-field entries of A and L, two FP64 products, and four outer iterations of every source
        total["bytes"] += 3 * bj + 4 * b
        total["flops"] += 240.0 * near + r * (2 * fj + 4 * f)
    return total


# ------------------------------------------------------------------ exact ----
# The collocation rule (flat triangles, centroids, r_c = 1.5 x the longest edge): the element's own entry and those
# within r_c by closed forms plus the 7-point rule on the smooth remainder, all others by the 3-point rule.
EXACT_MATVEC_MAX = 60000
EXACT_SOLVE_MAX = 6500


class _Dense:
    def __init__(self, verts, tris, k, beta):
        v = torch.tensor(np.asarray(verts), device="cuda")[torch.tensor(np.asarray(tris), device="cuda").long()]
        self.v, self.k = v, float(k)
        self.beta = None if beta is None else torch.tensor(beta, device="cuda")
        self.n = v.shape[0]
        self.c = v.sum(1) / 3.0
        cr = torch.linalg.cross(v[:, 1] - v[:, 0], v[:, 2] - v[:, 0])
        dbl = torch.linalg.vector_norm(cr, dim=1)
        self.area, self.normal = 0.5 * dbl, cr / dbl[:, None]
        edges = torch.stack([v[:, 1] - v[:, 0], v[:, 2] - v[:, 1], v[:, 0] - v[:, 2]])
        self.rc = 1.5 * float(torch.linalg.vector_norm(edges, dim=-1).max())
        b3 = torch.full((3, 3), 1.0 / 6.0, dtype=torch.float64, device="cuda") + 0.5 * torch.eye(
            3, dtype=torch.float64, device="cuda")
        self.q3 = torch.einsum("qv,nvd->qnd", b3, v).contiguous()
        s15 = math.sqrt(15.0)
        a, b = (6.0 - s15) / 21.0, (6.0 + s15) / 21.0
        rows = [[1 / 3, 1 / 3, 1 / 3]]
        for t in (a, b):
            rows += [[t, t, 1 - 2 * t], [t, 1 - 2 * t, t], [1 - 2 * t, t, t]]
        self.b7 = torch.tensor(rows, dtype=torch.float64, device="cuda")
        self.w7 = torch.tensor([9 / 40] + [(155 - s15) / 1200] * 3 + [(155 + s15) / 1200] * 3, dtype=torch.float64,
                               device="cuda")

    def _em1(self, kr):
        """e^{i kr} - 1 without cancellation."""
        h = torch.sin(0.5 * kr)
        return torch.complex(-2.0 * h * h, 2.0 * h * torch.cos(0.5 * kr))

    def _close(self, x, j):
        """L and M entries of points x close to elements j, pair by pair."""
        v, n, area = self.v[j], self.normal[j], self.area[j]
        d = ((x - v[:, 0]) * n).sum(-1)
        foot = x - d[:, None] * n
        ad = d.abs()
        inv_r = torch.zeros_like(d)
        for e in range(3):
            p, q = v[:, e], v[:, (e + 1) % 3]
            t = q - p
            le = torch.linalg.vector_norm(t, dim=-1)
            t = t / le[:, None]
            m = torch.linalg.cross(t, n)
            lo, hi = ((p - foot) * t).sum(-1), ((q - foot) * t).sum(-1)
            dist = ((p - foot) * m).sum(-1)
            r0 = torch.sqrt(dist * dist + d * d)
            rs = torch.maximum(r0, 1e-30 * le)
            inv_r += dist * (torch.asinh(hi / rs) - torch.asinh(lo / rs))
            for sign, l in ((1.0, hi), (-1.0, lo)):
                inv_r -= sign * ad * torch.atan2(dist * l, r0 * r0 + ad * torch.sqrt(r0 * r0 + l * l))
        r = [v[:, e] - x for e in range(3)]
        a = [torch.linalg.vector_norm(t, dim=-1) for t in r]
        num = (r[0] * torch.linalg.cross(r[1], r[2])).sum(-1)
        den = (a[0] * a[1] * a[2] + (r[0] * r[1]).sum(-1) * a[2] + (r[0] * r[2]).sum(-1) * a[1]
               + (r[1] * r[2]).sum(-1) * a[0])
        omega = 2.0 * torch.atan2(num, den)
        y = torch.einsum("qv,nvd->nqd", self.b7, v) - x[:, None, :]
        rad = torch.linalg.vector_norm(y, dim=-1)
        kr = self.k * rad
        em1 = self._em1(kr)
        f = 1j * kr * torch.polar(torch.ones_like(kr), kr) - em1
        smooth_l = (self.w7 * em1 / rad).sum(-1)
        smooth_m = (self.w7 * (y * n[:, None, :]).sum(-1) * f / rad ** 3).sum(-1)
        return (inv_r + area * smooth_l) / (4 * math.pi), (area * smooth_m - omega) / (4 * math.pi)

    def _own(self, j):
        """L entries of elements j at their own centroids."""
        v, c = self.v[j], self.c[j]
        total = torch.zeros(j.numel(), dtype=torch.complex128, device="cuda")
        for e in range(3):
            p, q = v[:, e], v[:, (e + 1) % 3]
            t = q - p
            le = torch.linalg.vector_norm(t, dim=-1)
            t = t / le[:, None]
            dist = ((p - c) * torch.linalg.cross(t, self.normal[j])).sum(-1)
            total += dist * (torch.asinh(((q - c) * t).sum(-1) / dist) - torch.asinh(((p - c) * t).sum(-1) / dist))
            sub = 0.5 * torch.linalg.vector_norm(torch.linalg.cross(p - c, q - c), dim=-1)
            y = torch.einsum("qv,vnd->nqd", self.b7, torch.stack([c, p, q])) - c[:, None, :]
            rad = torch.linalg.vector_norm(y, dim=-1)
            total += sub * (self.w7 * self._em1(self.k * rad) / rad).sum(-1)
        return total / (4 * math.pi)

    def rows(self, x, own=None):
        """(L, M) rows for points x; own: the element index whose centroid each point is, or None."""
        L = torch.zeros((x.shape[0], self.n), dtype=torch.complex128, device="cuda")
        M = torch.zeros_like(L)
        scale = self.area / (12.0 * math.pi)   # area x weight 1/3 over 4 pi
        for q in range(3):
            d = [self.q3[q, :, a][None, :] - x[:, a][:, None] for a in range(3)]
            rad = torch.sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2])
            kr = self.k * rad
            g = torch.polar(scale / rad, kr)
            L += g
            dn = (d[0] * self.normal[:, 0] + d[1] * self.normal[:, 1] + d[2] * self.normal[:, 2]) / (rad * rad)
            M += g * torch.complex(-dn, dn * kr)
        dist2 = sum((self.c[:, a][None, :] - x[:, a][:, None]) ** 2 for a in range(3))
        close = dist2 < self.rc * self.rc
        if own is not None:
            at = torch.arange(own.numel(), device="cuda")
            close[at, own] = False
        i, j = torch.nonzero(close, as_tuple=True)
        if i.numel():
            L[i, j], M[i, j] = self._close(x[i], j)
        if own is not None:
            L[at, own] = self._own(own)
            M[at, own] = 0.0
        return L, M

    def system_rows(self, own):
        """Rows of A = 1/2 + M - i k L diag(beta) and of L at the centroids of elements `own`."""
        L, M = self.rows(self.c[own], own)
        A = M - (1j * self.k) * L * self.beta[None, :]
        A[torch.arange(own.numel(), device="cuda"), own] += 0.5
        return A, L

    def chunks(self):
        step = max(16, min(1024, 25_000_000 // self.n))
        for a in range(0, self.n, step):
            yield torch.arange(a, min(self.n, a + step), device="cuda")

    def product(self, x):
        out = torch.empty_like(x)
        for own in self.chunks():
            A, _ = self.system_rows(own)
            out[..., own] = (A @ x.T).T if x.dim() == 2 else A @ x
        return out

    def monopole(self, src):
        """Boundary data -(d psi_in/dn - i k beta psi_in) of a monopole at the centroids."""
        r = self.c - torch.tensor(np.asarray(src), device="cuda")
        rad = torch.linalg.vector_norm(r, dim=-1)
        g = torch.polar(1.0 / (4 * math.pi * rad), self.k * rad)
        dn = (r * self.normal).sum(-1) / (rad * rad) * torch.complex(-torch.ones_like(rad), self.k * rad) * g
        return 1j * self.k * self.beta * g - dn

    def solve(self, src):
        """Solutions of A x = L gamma for every source, as rows."""
        A = torch.empty((self.n, self.n), dtype=torch.complex128, device="cuda")
        gamma = torch.stack([self.monopole(p) for p in src], 1)
        b = torch.empty_like(gamma)
        for own in self.chunks():
            A[own], L = self.system_rows(own)
            b[own] = L @ gamma
        return torch.linalg.solve(A, b).T.contiguous()


def _dense(case, seed, freq=None):
    beta_wall, src, rec = _inputs(case, seed)
    verts, tris, wall = _mesh_of(case, freq)
    d = _Dense(verts, tris, W.wavenumber(freq or case["freq"]), beta_wall[wall].astype(np.complex128))
    return d, src, rec


def exact(case, seed):
    kind = case["kind"]
    if kind == "sweep":
        out = []
        for f in np.geomspace(case["freq"], case["freq_hi"], int(case["jobs"])):
            d, src, _ = _dense(case, seed, f)
            out.append(d.solve(src) if d.n <= EXACT_SOLVE_MAX else None)
        return None if all(x is None for x in out) else out
    d, src, rec = _dense(case, seed)
    if kind == "solve":
        return d.solve(src)[0] if d.n <= EXACT_SOLVE_MAX else None
    if kind == "field":
        gamma = d.monopole(src[0])
        psi = d.monopole(src[0] + np.array([0.05, -0.04, 0.03])) / d.k
        q = gamma + 1j * d.k * d.beta * psi
        x = torch.tensor(rec, device="cuda")
        out = torch.empty(x.shape[0], dtype=torch.complex128, device="cuda")
        for a in range(0, x.shape[0], 64):
            L, M = d.rows(x[a:a + 64])
            out[a:a + 64] = L @ q - M @ psi
        rad = torch.linalg.vector_norm(x - torch.tensor(src[0], device="cuda"), dim=-1)
        return out + torch.polar(1.0 / (4 * math.pi * rad), d.k * rad)
    # products: the inner operator is a low-accuracy one on purpose (tens of percent off the dense matrix)
    if case["precision"] == "mixed16" or d.n > EXACT_MATVEC_MAX:
        return None
    rows = int(case.get("nrhs", 1))
    x = _rough_vectors(seed, d.n, rows)
    gamma = d.monopole(src[0])
    x += gamma * (math.sqrt(d.n) / torch.linalg.vector_norm(gamma))
    if kind != "multi":
        x = x[0]
    y = d.product(x)
    return [y, None] if kind == "setup" else y
