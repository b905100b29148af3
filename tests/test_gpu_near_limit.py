"""The near field where a leaf's columns and coefficients fill shared memory:
13,624 columns + 30^2 coefficients are 14,524 complex FP64 values of the
14,528 (227 KB) that a CTA may hold; one order more does not fit and is
refused.  The mixed product, half as wide, is the reference (1e-5)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_16073_gb300 as fb
from _cases import rel, seeded_vector
from paper_2103_16073_gb300 import workloads as W


def test_largest_leaf_block_that_fits():
    verts, tris, _ = W.shoebox_mesh(1.0, 0.9, 0.12, 72, 71, 8)
    n = tris.shape[0]
    mesh = fb.fb_mesh_create(verts, tris)
    fb.fb_mesh_set_admittance(mesh, np.full(n, 0.2, dtype=np.complex128))
    tree = fb.fb_tree_build(mesh, 40000)
    size, u = np.diff(fb.fb_tree_export(tree, 1)), fb.fb_tree_export(tree, 3)
    assert np.bincount(u[:, 0], weights=size[u[:, 1]]).max() == 13624
    x = torch.tensor(seeded_vector(n, 11), device="cuda")
    ops = []
    try:
        for prec, p in ((fb.FB_PREC_MIXED_FMM, 30), (fb.FB_PREC_FP64_FMM, 30), (fb.FB_PREC_FP64_FMM, 31)):
            ops.append(fb.fb_operator_create(mesh, tree, 60.0, fb.FB_OP_A, prec, 0.5, p))
        y = [fb.fb_operator_apply(op, x, torch.empty_like(x)).cpu().numpy() for op in ops[:2]]
        assert rel(y[1], y[0]) < 1e-5
        with pytest.raises(fb.FBError):
            fb.fb_operator_apply(ops[2], x, torch.empty_like(x))
    finally:
        for op in ops:
            fb.fb_operator_destroy(op)
        fb.fb_tree_destroy(tree)
        fb.fb_mesh_destroy(mesh)
