"""A call that the device refuses (here: a leaf block larger than shared
memory) reports its error and leaves nothing behind: the calls after it
succeed, on the same and on other objects."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_16073_gb300 as fb
from _cases import seeded_vector
from paper_2103_16073_gb300 import workloads as W


def test_calls_after_a_refused_one_succeed():
    verts, tris, _ = W.shoebox_mesh(1.0, 0.9, 0.12, 72, 71, 8)
    n = tris.shape[0]
    mesh = fb.fb_mesh_create(verts, tris)
    fb.fb_mesh_set_admittance(mesh, np.full(n, 0.2, dtype=np.complex128))
    tree = fb.fb_tree_build(mesh, 40000)   # leaf blocks of up to 13,624 columns
    x = torch.tensor(seeded_vector(n, 12), device="cuda")
    y = torch.empty_like(x)
    op = fb.fb_operator_create(mesh, tree, 60.0, fb.FB_OP_A, fb.FB_PREC_FP64_FMM, 0.5, 31)
    op32 = fb.fb_operator_create(mesh, tree, 60.0, fb.FB_OP_A, fb.FB_PREC_MIXED_FMM, 0.5, 30)
    try:
        for _ in range(2):
            with pytest.raises(fb.FBError) as e:
                fb.fb_operator_apply(op, x, y)
            assert e.value.code == 2   # FB_ERR_CUDA
            fb.fb_tree_destroy(fb.fb_tree_build(mesh, 40000))
            fb.fb_operator_apply(op32, x, y)
            assert bool(torch.isfinite(torch.view_as_real(y)).all())
    finally:
        fb.fb_operator_destroy(op)
        fb.fb_operator_destroy(op32)
        fb.fb_tree_destroy(tree)
        fb.fb_mesh_destroy(mesh)
