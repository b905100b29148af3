"""Block-Jacobi inverses on both sides of the line at 67 rows, the most that
are inverted in shared memory: trees whose largest leaf has 58 and 68 rows.  The reference solves with each
leaf's own block, read back from the operator; a solve and an inverse of a
well-conditioned block (identity plus compact) of 68 rows agree to 1e-11."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_16073_gb300 as fb
from _cases import rel, seeded_vector
from paper_2103_16073_gb300 import workloads as W


@pytest.mark.parametrize("name,most", [("shoebox", 68), ("lroom", 58)])
def test_blocks_on_both_sides_of_the_shared_memory_limit(name, most):
    if name == "shoebox":
        verts, tris, _ = W.shoebox_mesh(1.3, 1.1, 0.9, 17, 17, 13)
    else:
        verts, tris, _ = W.lroom_mesh(W.SOUND_SPEED / 150.0 / 8.0)
    n = tris.shape[0]
    mesh = fb.fb_mesh_create(verts, tris)
    fb.fb_mesh_set_admittance(mesh, np.full(n, 0.2, dtype=np.complex128))
    tree = fb.fb_tree_build(mesh, 70)
    op = fb.fb_operator_create(mesh, tree, 9.0, fb.FB_OP_A, fb.FB_PREC_FP64_FMM, 6.0, 12)
    pc = fb.fb_precond_create(op, fb.FB_PC_BLOCK_JACOBI)
    try:
        perm, start = fb.fb_tree_export(tree, 0), fb.fb_tree_export(tree, 1)
        u = fb.fb_tree_export(tree, 3)
        sizes = np.diff(start)
        assert sizes.max() == most and sizes.min() < 50
        v = seeded_vector(n, 79)
        z = torch.empty(n, dtype=torch.complex128, device="cuda")
        fb.fb_precond_apply(pc, torch.tensor(v, device="cuda"), z)
        z = z.cpu().numpy()
        for b in range(sizes.size):
            cols = [s for t, s in u if t == b]
            c0 = sum(sizes[s] for s in cols[:cols.index(b)])
            block = fb.fb_operator_export(op, 0, 0, b).reshape(sizes[b], -1)[:, c0:c0 + sizes[b]]
            rows = perm[start[b]:start[b + 1]]
            assert rel(z[rows], np.linalg.solve(block, v[rows])) < 1e-11, (b, sizes[b])
    finally:
        fb.fb_precond_destroy(pc)
        fb.fb_operator_destroy(op)
        fb.fb_tree_destroy(tree)
        fb.fb_mesh_destroy(mesh)
