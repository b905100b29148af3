"""Rounding errors of the element integrals against extended precision.  The
yardstick is the textbook form of each sum, evaluated in FP64 here on the
library's own centroids and normals: the device's error (root mean square over some thousand entries) may exceed it by
no more than 5 % (FMAs and another library move it by less)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_16073_gb300 as fb
from _cases import oracle_mesh, seeded_vector, workload

LD = np.longdouble
PI = LD("3.14159265358979323846264338327950288")


def dot(a, b):
    return (a * b).sum(-1)


def geometry(name):
    """(workload, corners, centroids, normals, areas) in extended precision."""
    wl = workload(name)
    v = wl.verts.astype(LD)[wl.tris]
    cr = np.cross(v[:, 1] - v[:, 0], v[:, 2] - v[:, 0])
    dbl = np.sqrt(dot(cr, cr))
    return wl, v, v.sum(1) / 3, cr / dbl[:, None], dbl / 2


def int_inv_r(x, v, nn):
    """int 1/R over flat triangles in the precision of the arguments, by differences of asinh and atan2."""
    d = dot(x - v[:, 0], nn)
    x0, ad, out = x - d[:, None] * nn, abs(d), np.zeros_like(d)
    for e in range(3):
        p, q = v[:, e], v[:, (e + 1) % 3]
        t = q - p
        t = t / np.sqrt(dot(t, t))[:, None]
        lm, lp, P = dot(p - x0, t), dot(q - x0, t), dot(p - x0, np.cross(t, nn))
        R0 = np.sqrt(P * P + d * d)
        Rm, Rp = np.sqrt(R0 * R0 + lm * lm), np.sqrt(R0 * R0 + lp * lp)
        out += P * (np.arcsinh(lp / R0) - np.arcsinh(lm / R0))
        out -= ad * (np.arctan2(P * lp, R0 * R0 + ad * Rp) - np.arctan2(P * lm, R0 * R0 + ad * Rm))
    return out


def smooth(k, x, v, area):
    """int (e^{ikR} - 1) / R by the seven-point rule, in the precision of the arguments."""
    T = x.dtype.type
    s = np.sqrt(T(15))
    rows, wt = [[T(1) / 3] * 3], [T(9) / 40] + [(155 - s) / 1200] * 3 + [(155 + s) / 1200] * 3
    for t in ((6 - s) / 21, (6 + s) / 21):
        rows += [[t, t, 1 - 2 * t], [t, 1 - 2 * t, t], [1 - 2 * t, t, t]]
    y = np.einsum("qv,nvd->nqd", np.array(rows), v) - x[:, None, :]
    R = np.sqrt(dot(y, y))
    h = np.sin(T(k) * R / 2)
    e1 = -2 * h * h + 1j * (2 * h * np.cos(T(k) * R / 2))
    return area * (np.array(wt) * e1 / R).sum(1)


def rms(e):
    return float(np.sqrt(np.mean(np.abs(e) ** 2)))


def test_closed_form_entries():
    """Single-layer entries within r_c at a wavenumber where the closed form is all but the whole."""
    wl, v, c, n, area = geometry("sub")
    k, rc = 2.0, oracle_mesh("sub").rc
    mesh = fb.fb_mesh_create(wl.verts, wl.tris)
    tree = fb.fb_tree_build(mesh, 64)
    op = fb.fb_operator_create(mesh, tree, k, fb.FB_OP_L, fb.FB_PREC_FP64_FMM, 0.5, 12)
    xc, xn = fb.fb_mesh_geometry(mesh)
    got, I, J = [], [], []
    try:
        perm, start, u = (fb.fb_tree_export(tree, w) for w in (0, 1, 3))
        for b in range(0, start.size - 1, 8):
            rows = perm[start[b]:start[b + 1]]
            cols = np.concatenate([perm[start[s]:start[s + 1]] for t, s in u if t == b])
            i, j = (a.ravel() for a in np.meshgrid(rows, cols, indexing="ij"))
            d = (c[i] - c[j]).astype(float)
            near = (dot(d, d) < rc * rc) & (i != j)
            got.append(fb.fb_operator_export(op, 0, 0, b)[near])
            I.append(i[near])
            J.append(j[near])
    finally:
        fb.fb_operator_destroy(op)
        fb.fb_tree_destroy(tree)
        fb.fb_mesh_destroy(mesh)
    got, I, J = np.concatenate(got), np.concatenate(I), np.concatenate(J)
    assert I.size > 5000
    exact = (int_inv_r(c[I], v[J], n[J]) + smooth(k, c[I], v[J], area[J])) / (4 * PI)
    x, n, v, area = xc[I], xn[J], v[J].astype(float), area[J].astype(float)
    plain = (int_inv_r(x, v, n) + smooth(k, x, v, area)) / (4 * np.pi)
    assert rms((got - exact) / exact) < 1.05 * rms((plain - exact) / exact)


def gauss(v):
    T = v.dtype.type
    b = [[T(2) / 3 if i == q else T(1) / 6 for i in range(3)] for q in range(3)]
    return np.stack([sum(w * v[:, i] for i, w in enumerate(r)) for r in b], 1)


def field(k, x, y, c, n, area, beta, psi, gam, rc):
    """L q - M psi at the points x by the three-point rule, elements within r_c left out."""
    out = []
    for r in x:
        d = y - r
        R = np.sqrt(dot(d, d))
        e = np.cos(k * R) + 1j * np.sin(k * R)
        w = (area / 3)[:, None] / (4 * np.pi if R.dtype == float else 4 * PI)
        L = (w * e / R).sum(1)
        M = (w * dot(n[:, None, :], d) / R ** 3 * (e * (-1 + 1j * k * R))).sum(1)
        z = L * (gam + 1j * k * beta * psi) - M * psi
        out.append(z[dot(c - r, c - r) >= rc * rc].sum())
    return np.array(out)


def test_receivers_at_a_low_wavenumber():
    """Receivers farther than r_c from every wall, where k R stays small and its rounding does not dominate."""
    wl, v, c, n, area = geometry("sub")
    k, rc = 2.0, oracle_mesh("sub").rc
    rng = np.random.default_rng(5)
    x = rc + (np.array(wl.room) - 2 * rc) * rng.uniform(0.0, 1.0, size=(400, 3))
    psi, gam = seeded_vector(wl.n, 1), seeded_vector(wl.n, 2)
    mesh = fb.fb_mesh_create(wl.verts, wl.tris)
    fb.fb_mesh_set_admittance(mesh, wl.beta)
    try:
        xc, xn = fb.fb_mesh_geometry(mesh)
        out = torch.empty(400, dtype=torch.complex128, device="cuda")
        got = fb.fb_eval_field(mesh, k, *(torch.tensor(a, device="cuda") for a in (psi, gam, x)), out).cpu().numpy()
    finally:
        fb.fb_mesh_destroy(mesh)
    rest = (wl.beta, psi, gam, rc)
    exact = field(LD(k), x.astype(LD), gauss(v), c, n, area, *rest)
    plain = field(k, x, gauss(v.astype(float)), xc, xn, area.astype(float), *rest)
    assert rms(got - exact) < 1.05 * rms(plain - exact)
