"""Staging buffers of the staged passes for several right-hand sides: the
autotuner times staged forms in the batches that the product runs them in,
buffers that hold some but not all right-hand sides (batches with a
remainder), and buffers that grow after a graph was captured with the old
ones.  A right-hand side's result does not depend on its batch beyond the
order of the scattered additions: FP64 to 1e-12, FP32 to 1e-5."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_16073_gb300 as fb
from _cases import rel, seeded_vector, workload

STAGED = [4 | 8] * 13
TENSOR = [4 | 8 | 16 | 32 | 1024 | 2048] * 13


@pytest.fixture(scope="module")
def sub():
    wl = workload("sub")
    mesh = fb.fb_mesh_create(wl.verts, wl.tris)
    fb.fb_mesh_set_admittance(mesh, wl.beta)
    tree = fb.fb_tree_build(mesh, 64)
    yield wl, mesh, tree
    fb.fb_tree_destroy(tree)
    fb.fb_mesh_destroy(mesh)


def vectors(wl, n):
    return torch.tensor(np.stack([seeded_vector(wl.n, 120 + r) for r in range(n)]), device="cuda")


def multi(op, X):
    Y = torch.empty_like(X)
    fb.fb_operator_apply_multi(op, X, Y)
    torch.cuda.synchronize()
    return Y.cpu().numpy()


def tune_launches(sub, prec, nrhs):
    wl, mesh, tree = sub
    op = fb.fb_operator_create(mesh, tree, 18.0, fb.FB_OP_A, prec, 0.5, 24)
    try:
        before = fb.fb_kernel_launches()
        fb.fb_operator_autotune(op, nrhs)
        return fb.fb_kernel_launches() - before
    finally:
        fb.fb_operator_destroy(op)


@pytest.mark.parametrize("prec", [fb.FB_PREC_FP64_FMM, fb.FB_PREC_MIXED_FMM])
def test_autotuner_times_staged_forms_in_one_batch(sub, prec):
    """Every candidate is launched the same number of times whatever the
    number of right-hand sides (three of 8,928 pairs x 576 coefficients fit
    one batch); only the plans of the forms chosen in the end may differ by
    some launches.  A launch per right-hand side would make the staged
    candidates, most of all launches, three times as many."""
    assert tune_launches(sub, prec, 3) < 1.5 * tune_launches(sub, prec, 1)


@pytest.mark.parametrize("prec,forms,tol", [(fb.FB_PREC_FP64_FMM, STAGED, 1e-12),
                                            (fb.FB_PREC_MIXED_FMM, STAGED, 1e-5),
                                            (fb.FB_PREC_MIXED_FMM, TENSOR, 1e-5)])
def test_batches_with_a_remainder(sub, prec, forms, tol):
    """Order 30 on the leaf level: 8,928 pairs x 900 coefficients are 61 MiB in
    FP32 and 123 MiB in FP64, so 256 MiB hold four or two of seven."""
    wl, mesh, tree = sub
    assert fb.fb_tree_export(tree, 4, 3).shape[0] == 8928
    X = vectors(wl, 7)
    op = fb.fb_operator_create(mesh, tree, 18.0, fb.FB_OP_A, prec, 0.5, 30)
    try:
        fb.fb_operator_set_forms(op, forms)
        one = np.concatenate([multi(op, X[r:r + 1].contiguous()) for r in range(7)])
        assert rel(multi(op, X), one) < tol
    finally:
        fb.fb_operator_destroy(op)


@pytest.mark.parametrize("prec,forms,tol", [(fb.FB_PREC_FP64_FMM, STAGED, 1e-12),
                                            (fb.FB_PREC_MIXED_FMM, TENSOR, 1e-5)])
def test_buffers_that_grow_after_a_capture(sub, prec, forms, tol):
    wl, mesh, tree = sub
    X = vectors(wl, 5)
    op = fb.fb_operator_create(mesh, tree, 18.0, fb.FB_OP_A, prec, 0.5, 16)
    try:
        fb.fb_operator_set_forms(op, forms)
        ref = np.concatenate([multi(op, X[r:r + 1].contiguous()) for r in range(5)])
        fb.fb_operator_use_graphs(op, True)
        for n in (1, 2, 5, 2, 1):
            assert rel(multi(op, X[:n].contiguous()), ref[:n]) < tol
    finally:
        fb.fb_operator_destroy(op)
