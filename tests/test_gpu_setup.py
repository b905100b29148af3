"""Setup kernels at the edges of their splits.

Near-field blocks (128 columns and 32 rows per CTA, closed-form entries
collected apart) of every operator kind against rows of the dense operator,
which integrates entry by entry: the same rule in FP64, so 1e-12 of the
block's largest entry (a few hundred roundings).  P2M / L2P rows at an order
whose work array no longer fits shared memory against a small order's:
leading degrees do not depend on the order, and the downward Bessel
recurrence started higher differs by rounding only (1e-12 of each degree's
largest entry).  Coaxial sets on both sides of k t = 1 through the whole
product against the dense operator (the FMM's truncation, 1e-5)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_16073_gb300 as fb
from _cases import rel, seeded_vector, workload


@pytest.fixture(scope="module")
def ragged():
    wl = workload("ragged")
    mesh = fb.fb_mesh_create(wl.verts, wl.tris)
    fb.fb_mesh_set_admittance(mesh, wl.beta)
    tree = fb.fb_tree_build(mesh, 64)
    yield wl, mesh, tree
    fb.fb_tree_destroy(tree)
    fb.fb_mesh_destroy(mesh)


@pytest.mark.parametrize("kind", [fb.FB_OP_L, fb.FB_OP_M, fb.FB_OP_LP, fb.FB_OP_A, fb.FB_OP_MP])
def test_near_blocks_equal_dense_rows(ragged, kind):
    wl, mesh, tree = ragged
    perm, start = fb.fb_tree_export(tree, 0), fb.fb_tree_export(tree, 1)
    u = fb.fb_tree_export(tree, 3)
    op = fb.fb_operator_create(mesh, tree, wl.k, kind, fb.FB_PREC_FP64_FMM, 6.0, 14)
    dense = fb.fb_operator_create(mesh, tree, wl.k, kind, fb.FB_PREC_FP64_DENSE)
    try:
        nleaf = start.size - 1
        widths = [sum(start[s + 1] - start[s] for t, s in u if t == b) for b in range(nleaf)]
        for b in {0, nleaf - 1, int(np.argmax(widths)), int(np.argmax(np.diff(start)))}:
            rows = perm[start[b]:start[b + 1]]
            cols = np.concatenate([perm[start[s]:start[s + 1]] for t, s in u if t == b])
            got = fb.fb_operator_export(op, 0, 0, b).reshape(rows.size, cols.size)
            want = np.stack([fb.fb_operator_export(dense, 6, 0, int(i))[cols] for i in rows])
            assert np.max(np.abs(got - want)) < 1e-12 * np.max(np.abs(want)), (kind, b)
    finally:
        fb.fb_operator_destroy(op)
        fb.fb_operator_destroy(dense)


@pytest.mark.parametrize("kind", [fb.FB_OP_A, fb.FB_OP_LP])
def test_p2m_leading_degrees_do_not_depend_on_the_order(ragged, kind):
    wl, mesh, tree = ragged
    k, q = 300.0, 24
    rows = {}
    for p in (151, 160):   # the last order with shared-memory work arrays is 150
        op = fb.fb_operator_create(mesh, tree, k, kind, fb.FB_PREC_FP64_FMM, 0.1, p)
        try:
            P = int(fb.fb_operator_info(op)[2][-1])
            rows[p] = [fb.fb_operator_export(op, w, 0, 0).reshape(-1, P * P)[:, :q * q] for w in (1, 2)]
        finally:
            fb.fb_operator_destroy(op)
    low = fb.fb_operator_create(mesh, tree, 5.0, kind, fb.FB_PREC_FP64_FMM, 0.1, q)
    low2 = fb.fb_operator_create(mesh, tree, 5.0, kind, fb.FB_PREC_FP64_FMM, 0.1, 40)
    try:
        for w in (0, 1):
            a = fb.fb_operator_export(low, w + 1, 0, 0).reshape(-1, q * q)
            b = fb.fb_operator_export(low2, w + 1, 0, 0).reshape(-1, 1600)[:, :q * q]
            for x, y in ((a, b), (rows[151][w], rows[160][w])):
                for n in range(q):
                    s = slice(n * n, (n + 1) ** 2)
                    assert np.max(np.abs(x[:, s] - y[:, s])) <= 1e-12 * np.max(np.abs(y[:, s])), (w, n)
    finally:
        fb.fb_operator_destroy(low)
        fb.fb_operator_destroy(low2)


@pytest.mark.parametrize("k", [0.4, 3.0])
def test_product_on_both_sides_of_unit_translation_distance(ragged, k):
    wl, mesh, tree = ragged
    x = torch.tensor(seeded_vector(wl.n, 5), device="cuda")
    y = []
    for prec in (fb.FB_PREC_FP64_FMM, fb.FB_PREC_FP64_DENSE):
        op = fb.fb_operator_create(mesh, tree, k, fb.FB_OP_A, prec)
        try:
            y.append(fb.fb_operator_apply(op, x, torch.empty_like(x)).cpu().numpy())
        finally:
            fb.fb_operator_destroy(op)
    assert rel(y[0], y[1]) < 1e-5
