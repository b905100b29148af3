"""Per-pair translation tiles at the orders where shared memory holds one or
two columns of a tile (16-byte types: one from order 69, FP32: two from 77,
one from 99), up to the largest that fit, and M2M into a level whose order no
longer does (53 -> 90 in the 16-byte types), which runs staged instead.  The
staged passes compute the same sums in other kernels and are the reference.

Tolerances: rounding of three steps of sums of at most p <= 104 terms, growing
like their square root: FP64 (1.1e-16) stays below 1e-12, double-FP32 (2^-48)
below 1e-11, FP32 (6e-8) below 3 p 6e-8 < 2e-5."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_16073_gb300 as fb
from _cases import rel, seeded_vector, workload

TILES, TILES_DF, STAGED = [0] * 13, [256 | 512] * 13, [4 | 8] * 13
# (wavenumber, d0, orders of levels 2 and 3)
ORDERS = [(100.0, 0.5, (70, 37)), (115.0, 0.5, (80, 42)), (101.0, 6.0, (90, 52)), (105.0, 6.0, (93, 54)),
          (120.0, 6.0, (104, 60))]


@pytest.fixture(scope="module")
def sub():
    wl = workload("sub")
    mesh = fb.fb_mesh_create(wl.verts, wl.tris)
    fb.fb_mesh_set_admittance(mesh, wl.beta)
    tree = fb.fb_tree_build(mesh, 64)
    yield wl, mesh, tree
    fb.fb_tree_destroy(tree)
    fb.fb_mesh_destroy(mesh)


def apply(op, X):
    Y = torch.empty_like(X)
    (fb.fb_operator_apply if X.dim() == 1 else fb.fb_operator_apply_multi)(op, X, Y)
    torch.cuda.synchronize()
    return Y.cpu().numpy()


@pytest.mark.parametrize("nrhs", [1, 3])
@pytest.mark.parametrize("k,d0,orders", ORDERS)
def test_high_order_tiles_equal_staged(sub, k, d0, orders, nrhs):
    wl, mesh, tree = sub
    X = torch.tensor(np.stack([seeded_vector(wl.n, 40 + r) for r in range(nrhs)]), device="cuda")
    X = X[0].contiguous() if nrhs == 1 else X
    op = fb.fb_operator_create(mesh, tree, k, fb.FB_OP_A, fb.FB_PREC_FP64_FMM, d0, 12)
    op32 = fb.fb_operator_create(mesh, tree, k, fb.FB_OP_A, fb.FB_PREC_MIXED_FMM, d0, 12)
    try:
        assert tuple(fb.fb_operator_info(op)[2][2:4]) == orders
        fb.fb_operator_set_forms(op, STAGED)
        ref = apply(op, X)
        for forms, tol in ((TILES, 1e-12), (TILES_DF, 1e-11)):
            fb.fb_operator_set_forms(op, forms)
            assert rel(apply(op, X), ref) < tol
        fb.fb_operator_set_forms(op32, TILES)
        assert rel(apply(op32, X), ref) < 2e-5
    finally:
        fb.fb_operator_destroy(op)
        fb.fb_operator_destroy(op32)
