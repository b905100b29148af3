"""Double-FP32 tiles on values outside FP32's normal range.  A product is
linear, so scaling its input by a power of two scales its output exactly in
FP64; in double-FP32 the leaf multipoles of a vector scaled so that the
largest is 2^-130 are subnormal (spacing 2^-149, 2^-19 of the largest), which
leaves the product good to 1e-3.  Flushed to zero they would take the leaf
level's far field with them."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_16073_gb300 as fb
from _cases import rel, seeded_vector, workload


def test_subnormal_expansions():
    wl = workload("sub")
    mesh = fb.fb_mesh_create(wl.verts, wl.tris)
    fb.fb_mesh_set_admittance(mesh, wl.beta)
    tree = fb.fb_tree_build(mesh, 64)
    op = fb.fb_operator_create(mesh, tree, 18.0, fb.FB_OP_A, fb.FB_PREC_FP64_FMM, 0.5, 12)
    try:
        P = int(fb.fb_operator_info(op)[2][-1]) ** 2
        perm, start = fb.fb_tree_export(tree, 0), fb.fb_tree_export(tree, 1)
        v = seeded_vector(wl.n, 33)
        W = np.concatenate([fb.fb_operator_export(op, 1, 0, b).reshape(-1, P) for b in range(start.size - 1)])
        leaf = np.add.reduceat(W * v[perm][:, None], start[:-1], axis=0)
        s = 2.0 ** (-130 - np.ceil(np.log2(np.max(np.abs(leaf)))))
        x = torch.tensor(v * s, device="cuda")
        y = []
        for forms in (0, 256 | 512):
            fb.fb_operator_set_forms(op, [forms] * 13)
            y.append(fb.fb_operator_apply(op, x, torch.empty_like(x)).cpu().numpy() / s)
        fb.fb_operator_set_forms(op, [0] * 13)
        big = fb.fb_operator_apply(op, torch.tensor(v, device="cuda"), torch.empty_like(x)).cpu().numpy()
        assert rel(y[0], big) < 1e-12
        assert rel(y[1], big) < 1e-3
    finally:
        fb.fb_operator_destroy(op)
        fb.fb_tree_destroy(tree)
        fb.fb_mesh_destroy(mesh)
