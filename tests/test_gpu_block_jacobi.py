"""Block-Jacobi inverses at the edges of their kernel: blocks of a few rows,
around the 66 rows that fit shared memory, and larger ones in global memory,
against a direct solve with the oracle's leaf blocks.

Tolerance: the entries agree to the 1e-10 of the element integrals, and the
blocks (identity plus compact, at most 400 rows) are well conditioned."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_16073_gb300 as fb
from _cases import oracle_dense, oracle_mesh, rel, seeded_vector, workload
from oracle import learned
from oracle.octree import Octree


@pytest.mark.parametrize("leaf", [4, 30, 64, 70, 400])
def test_block_jacobi_against_oracle(leaf):
    wl = workload("small")
    mesh = fb.fb_mesh_create(wl.verts, wl.tris)
    fb.fb_mesh_set_admittance(mesh, wl.beta)
    tree = fb.fb_tree_build(mesh, leaf)
    op = fb.fb_operator_create(mesh, tree, wl.k, fb.FB_OP_A, fb.FB_PREC_FP64_FMM, 6.0, 12)
    pc = fb.fb_precond_create(op, fb.FB_PC_BLOCK_JACOBI)
    try:
        v = seeded_vector(wl.n, 78)
        z = torch.empty(wl.n, dtype=torch.complex128, device="cuda")
        fb.fb_precond_apply(pc, torch.tensor(v, device="cuda"), z)
        torch.cuda.synchronize()
        om = oracle_mesh("small")
        el = om.el
        T = learned.TreeInfo(Octree(np.concatenate([el.v0, el.v1, el.v2]), el.centroid, om.rc, leaf))
        A = oracle_dense("small")["A"]
        assert rel(z.cpu().numpy(), learned.block_jacobi(lambda i, j: A[np.ix_(i, j)], T, v)) < 1e-8
    finally:
        fb.fb_precond_destroy(pc)
        fb.fb_operator_destroy(op)
        fb.fb_tree_destroy(tree)
        fb.fb_mesh_destroy(mesh)
