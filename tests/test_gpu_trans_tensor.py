"""Composed translations on the tensor cores at the edges of their tiles: row
blocks of 2 p^2 rows around one, two and three tiles of at most 224, odd
orders (targets that allow 8-byte adds only), pair counts below and above the
128 of a tile, levels with fewer matrices than a cluster has CTAs, and several
right-hand sides.  The per-pair tiles in FP64 are the reference.

Tolerance: 3xTF32 drops products below 2^-21 of a term and sums in FP32, as
the FP32 tiles do; both stay below the 1e-5 of the mixed-precision operators."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_16073_gb300 as fb
from _cases import rel, seeded_vector, workload

# (wavenumber, p_min, leaf size); FP32 coefficients bound the order from above
# where boxes are small against the wavelength
CASES = [(1.0, p, leaf) for p in (1, 2, 3, 5, 10, 11) for leaf in (16, 200)]
CASES += [(18.0, p, 64) for p in (14, 15, 18, 19, 21)]


@pytest.fixture(scope="module")
def sub():
    wl = workload("sub")
    mesh = fb.fb_mesh_create(wl.verts, wl.tris)
    fb.fb_mesh_set_admittance(mesh, wl.beta)
    trees = {leaf: fb.fb_tree_build(mesh, leaf) for leaf in (16, 64, 200)}
    yield wl, mesh, trees
    for t in trees.values():
        fb.fb_tree_destroy(t)
    fb.fb_mesh_destroy(mesh)


def apply(op, X):
    Y = torch.empty_like(X)
    (fb.fb_operator_apply if X.dim() == 1 else fb.fb_operator_apply_multi)(op, X, Y)
    torch.cuda.synchronize()
    return Y.cpu().numpy()


@pytest.mark.parametrize("nrhs", [1, 3])
@pytest.mark.parametrize("k,pmin,leaf", CASES)
def test_tensor_equals_tiles(sub, k, pmin, leaf, nrhs):
    wl, mesh, trees = sub
    X = torch.tensor(np.stack([seeded_vector(wl.n, 80 + r) for r in range(nrhs)]), device="cuda")
    X = X[0].contiguous() if nrhs == 1 else X
    args = (mesh, trees[leaf], k, fb.FB_OP_A)
    op = fb.fb_operator_create(*args, fb.FB_PREC_FP64_FMM, 0.5, pmin)
    op32 = fb.fb_operator_create(*args, fb.FB_PREC_MIXED_FMM, 0.5, pmin)
    try:
        fb.fb_operator_set_forms(op, [0] * 13)
        ref = apply(op, X)
        fb.fb_operator_set_forms(op32, [1 | 2] * 13)
        assert rel(apply(op32, X), ref) < 1e-5
    finally:
        fb.fb_operator_destroy(op)
        fb.fb_operator_destroy(op32)
