"""P2M and the near field with L2P at the edges of their tiles: leaves of a few
and of more than 256 elements (chunks of the gather), orders above 256
coefficients and below a warp, odd column counts, rows split over CTAs, and
chunks of right-hand sides that are not full.  The kernels for one right-hand
side and for four are different instances and have to agree; the FP64 product
with another leaf size is the reference of both.

Tolerances: FP64 sums of at most 10^4 terms agree to 1e-12; expansions of this
accuracy (d0 = 6) to 1e-5 between trees; FP32 to 1e-5, 16-bit entries (relative
rounding 2^-9) to 2^-8."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_16073_gb300 as fb
from _cases import rel, seeded_vector, workload

NR = 5


@pytest.fixture(scope="module")
def sub():
    wl = workload("sub")
    mesh = fb.fb_mesh_create(wl.verts, wl.tris)
    fb.fb_mesh_set_admittance(mesh, wl.beta)
    X = torch.tensor(np.stack([seeded_vector(wl.n, 90 + r) for r in range(NR)]), device="cuda")
    yield mesh, X
    fb.fb_mesh_destroy(mesh)


def one(op, X):
    Y = torch.empty_like(X)
    for r in range(X.shape[0]):
        fb.fb_operator_apply(op, X[r].contiguous(), Y[r])
    torch.cuda.synchronize()
    return Y.cpu().numpy()


def multi(op, X):
    Y = torch.empty_like(X)
    fb.fb_operator_apply_multi(op, X, Y)
    torch.cuda.synchronize()
    return Y.cpu().numpy()


@pytest.mark.parametrize("k,leaf", [(18.0, 5), (18.0, 33), (18.0, 300), (18.0, 1100), (60.0, 64), (2.0, 20)])
def test_leaf_kernels(sub, k, leaf):
    mesh, X = sub
    tree, other = fb.fb_tree_build(mesh, leaf), fb.fb_tree_build(mesh, 64 if leaf != 64 else 100)
    args = (k, fb.FB_OP_A)
    op = fb.fb_operator_create(mesh, tree, *args, fb.FB_PREC_FP64_FMM, 6.0, 12)
    op32 = fb.fb_operator_create(mesh, tree, *args, fb.FB_PREC_MIXED_FMM, 6.0, 12)
    ref = fb.fb_operator_create(mesh, other, *args, fb.FB_PREC_FP64_FMM, 6.0, 12)
    try:
        y, y32 = one(op, X), one(op32, X)
        assert rel(y, one(ref, X)) < 1e-5
        assert rel(y32, y) < 1e-5
        for n in range(2, NR + 1):
            assert rel(multi(op, X[:n].contiguous()), y[:n]) < 1e-12
            assert rel(multi(op32, X[:n].contiguous()), y32[:n]) < 1e-5
        fb.fb_operator_set_near_bf16(op32, True)
        assert rel(one(op32, X), y) < 2.0**-8
        assert rel(multi(op32, X), y) < 2.0**-8
    finally:
        for o in (op, op32, ref):
            fb.fb_operator_destroy(o)
        for t in (tree, other):
            fb.fb_tree_destroy(t)
