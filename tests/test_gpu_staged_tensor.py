"""Staged translations on the tensor cores at the edges of their items: orders
around the multiples of 16 of a K chunk and a column block, above 64 (two row
blocks of the coaxial pass need more than one accumulator group) and above 128
(accumulators of 256 columns, fewest pipeline stages), polar-angle groups of a
few slots, with the coaxial pass on either kind of core, M2L and M2M / L2L,
and several right-hand sides.  The same passes in FP64 are the reference.

Tolerance: three steps of at most p^2 ~ 2 10^4 FP32 roundings of 6e-8 that
grow like their square root, 3 p 6e-8 < 3e-5."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_16073_gb300 as fb
from _cases import rel, seeded_vector, workload

STAGED = [4 | 8] * 13
ROT = [4 | 8 | 16 | 32] * 13              # rotations on the tensor cores
ALL = [4 | 8 | 16 | 32 | 1024 | 2048] * 13   # ... and the coaxial pass
# (wavenumber, d0, p_min)
ORDERS = [(1.0, 0.5, 1), (1.0, 0.5, 2), (1.0, 0.5, 7), (18.0, 0.5, 15), (18.0, 0.5, 16), (18.0, 0.5, 17),
          (60.0, 0.5, 33), (60.0, 0.5, 48), (60.0, 0.5, 49), (137.0, 6.0, 12), (170.0, 6.0, 12)]


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


@pytest.mark.parametrize("nrhs", [1, 2])
@pytest.mark.parametrize("k,d0,pmin", ORDERS)
def test_tensor_equals_fp64(sub, k, d0, pmin, nrhs):
    wl, mesh, tree = sub
    X = torch.tensor(np.stack([seeded_vector(wl.n, 70 + r) for r in range(nrhs)]), device="cuda")
    X = X[0].contiguous() if nrhs == 1 else X
    op = fb.fb_operator_create(mesh, tree, k, fb.FB_OP_A, fb.FB_PREC_FP64_FMM, d0, pmin)
    op32 = fb.fb_operator_create(mesh, tree, k, fb.FB_OP_A, fb.FB_PREC_MIXED_FMM, d0, pmin)
    try:
        fb.fb_operator_set_forms(op, STAGED)
        ref = apply(op, X)
        for forms in (ROT, ALL):
            fb.fb_operator_set_forms(op32, forms)
            assert rel(apply(op32, X), ref) < 3e-5
    finally:
        fb.fb_operator_destroy(op)
        fb.fb_operator_destroy(op32)
