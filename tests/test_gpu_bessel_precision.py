"""Spherical Bessel functions of the setup against extended precision.  Column
(0, 0) of the M2L matrix along z holds sqrt(2n+1) h_n(k tau) in its entries of
order 0 (the rotations are the identity but for their own rounding, which is
divided out), whose real part is j_n; degrees below k tau, where y_n is not
larger.  The yardstick is the downward recurrence
in FP64 with a division per step (3e-16); the device may have twice its error,
which covers a handful of roundings in the composed matrix."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_16073_gb300 as fb
from _cases import workload

P = 32
ALONG_Z = 3 * 49 + 3 * 7 + 3 + 2   # offset code of (0, 0, 2) box sides


def bessel(x, T):
    """j_n(x), n < P, by the downward recurrence in the type T."""
    x = x.astype(T)
    a, b = np.zeros_like(x), np.full_like(x, T(1e-280))
    out = []
    for n in range(P + 24 + int(x.max()), 0, -1):
        a, b = b, (2 * n + 1) / x * b - a
        out.append(b)
        big = np.abs(b) > 1e200
        for v in out[-P:] + [a]:
            v[big] *= T(1e-200)
        b = out[-1]
    out = np.stack(out[::-1][:P])
    j0, j1 = np.sin(x) / x, np.sin(x) / (x * x) - np.cos(x) / x
    return out * np.where(np.abs(j0) >= np.abs(j1), j0 / out[0], j1 / out[1])


def rms(a):
    return float(np.sqrt(np.mean(np.square(a.astype(float)))))


def test_translation_coefficients():
    wl = workload("sub")
    mesh = fb.fb_mesh_create(wl.verts, wl.tris)
    fb.fb_mesh_set_admittance(mesh, wl.beta)
    tree = fb.fb_tree_build(mesh, 64)
    ks = np.linspace(12.0, 40.0, 15)
    got = []
    try:
        side = fb.fb_tree_info(tree)[2]
        for k in ks:
            op = fb.fb_operator_create(mesh, tree, k, fb.FB_OP_L, fb.FB_PREC_FP64_FMM, 0.5, P)
            try:
                assert list(fb.fb_operator_info(op)[2][2:4]) == [P, P]
                T = fb.fb_operator_export(op, 3, 3, ALONG_Z).reshape(P * P, P * P)[:, 0]
                d = [fb.fb_operator_export(op, 8, n, ALONG_Z).reshape(2 * n + 1, -1)[n, n].real for n in range(P)]
            finally:
                fb.fb_operator_destroy(op)
            got.append([abs(T[n * n + n].real / (d[n] * d[0])) / np.sqrt(2 * n + 1) for n in range(P)])
    finally:
        fb.fb_tree_destroy(tree)
        fb.fb_mesh_destroy(mesh)
    x = ks * (2.0 * (side / 8))
    got, exact, plain = np.array(got).T, np.abs(bessel(x, np.longdouble)), np.abs(bessel(x, np.float64))
    scale = np.maximum(exact, np.roll(exact, 1, 0))   # a zero's neighbour sets the size
    inside = np.arange(P)[:, None] < x[None, :]
    err = [rms(((a - exact) / scale)[inside]) for a in (got, plain)]
    assert err[0] < 2.0 * err[1]
