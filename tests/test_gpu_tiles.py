"""Per-pair translation tiles at the edges of their row and column splits:
orders around the multiples at which a lane takes more rows (4, 8, 12 in
FP32, 4 to 8 in the 16-byte types) or a tile fewer columns, unequal orders
across M2M and L2L, ragged column counts and several right-hand sides.  The
staged passes compute the same sums in other kernels and are the reference;
their entries are pinned to the oracle in test_gpu_fmm.py and
test_gpu_staged.py.

Tolerances: FP64 rounding of sums of at most p^2 ~ 2,400 terms in three steps
stays below 1e-12; double-FP32 carries 2^-48 per step, below 1e-11; FP32
carries 6e-8 per step, below 1e-5."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_16073_gb300 as fb
from _cases import rel, seeded_vector, workload

TILES, TILES_DF, STAGED = [0] * 13, [256 | 512] * 13, [4 | 8] * 13
# (wavenumber, d0, p_min): at the small wavenumbers every level has order p_min
ORDERS = [(1.0, 0.5, 1), (1.0, 0.5, 2), (1.0, 0.5, 3), (1.0, 0.5, 4), (1.0, 0.5, 5), (4.0, 0.5, 8), (4.0, 0.5, 9),
          (18.0, 0.5, 2), (18.0, 0.5, 12), (18.0, 0.5, 13), (18.0, 0.5, 16), (18.0, 0.5, 17), (18.0, 0.5, 24),
          (18.0, 0.5, 25), (60.0, 0.5, 33), (60.0, 0.5, 49)]


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
@pytest.mark.parametrize("k,d0,pmin", ORDERS)
def test_tiles_equal_staged(sub, k, d0, pmin, nrhs):
    wl, mesh, tree = sub
    X = torch.tensor(np.stack([seeded_vector(wl.n, 60 + r) for r in range(nrhs)]), device="cuda")
    X = X[0].contiguous() if nrhs == 1 else X
    op = fb.fb_operator_create(mesh, tree, k, fb.FB_OP_A, fb.FB_PREC_FP64_FMM, d0, pmin)
    op32 = fb.fb_operator_create(mesh, tree, k, fb.FB_OP_A, fb.FB_PREC_MIXED_FMM, d0, pmin)
    try:
        fb.fb_operator_set_forms(op, STAGED)
        ref = apply(op, X)
        fb.fb_operator_set_forms(op, TILES)
        assert rel(apply(op, X), ref) < 1e-12
        fb.fb_operator_set_forms(op, TILES_DF)
        assert rel(apply(op, X), ref) < 1e-11
        fb.fb_operator_set_forms(op32, TILES)
        assert rel(apply(op32, X), ref) < 1e-5
    finally:
        fb.fb_operator_destroy(op)
        fb.fb_operator_destroy(op32)
