"""What the double-FP32 tiles hold in 64 bits: phases, sums and differences of
their load and store steps, as the staged passes do.  The arithmetic between
is the same 48-bit multiply-adds in both, so their errors against FP64 agree
to a few percent (the order of additions differs); phases of 48 bits would
add 7 to 17 %.  Bound: 1.04 over four vectors an order."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_16073_gb300 as fb
from _cases import rel, seeded_vector, workload

FP64, TILES_DF, STAGED_DF = 4 | 8, 256 | 512, 4 | 8 | 64 | 128


@pytest.mark.parametrize("k,p", [(18.0, 12), (18.0, 16), (18.0, 20), (60.0, 33), (60.0, 48)])
def test_error_is_that_of_the_staged_passes(k, p):
    wl = workload("sub")
    mesh = fb.fb_mesh_create(wl.verts, wl.tris)
    fb.fb_mesh_set_admittance(mesh, wl.beta)
    tree = fb.fb_tree_build(mesh, 64)
    op = fb.fb_operator_create(mesh, tree, k, fb.FB_OP_A, fb.FB_PREC_FP64_FMM, 0.5, p)
    try:
        err = []
        for r in range(4):
            x = torch.tensor(seeded_vector(wl.n, 200 + r), device="cuda")
            y = []
            for forms in (FP64, TILES_DF, STAGED_DF):
                fb.fb_operator_set_forms(op, [forms] * 13)
                y.append(fb.fb_operator_apply(op, x, torch.empty_like(x)).cpu().numpy())
            err.append((rel(y[1], y[0]), rel(y[2], y[0])))
        tiles, staged = np.sqrt(np.mean(np.square(err), axis=0))
        assert tiles < 1.04 * staged
    finally:
        fb.fb_operator_destroy(op)
        fb.fb_tree_destroy(tree)
        fb.fb_mesh_destroy(mesh)
