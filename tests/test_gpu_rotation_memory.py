"""Rotation data that a tree keeps: the FP64 real factors of every direction,
the complex blocks of the composed orders and the phases, nothing else; and
the exported factors of a mixed operator are the FP64 ones rounded to FP32."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_16073_gb300 as fb
from _cases import workload


def free_bytes():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_rotation_data_of_a_tree():
    wl = workload("sub")
    mesh = fb.fb_mesh_create(wl.verts, wl.tris)
    fb.fb_mesh_set_admittance(mesh, wl.beta)
    tree = fb.fb_tree_build(mesh, 64)
    ops = []
    try:
        free = [free_bytes()]
        for prec in (fb.FB_PREC_MIXED_FMM, fb.FB_PREC_MIXED_FMM, fb.FB_PREC_FP64_FMM):
            ops.append(fb.fb_operator_create(mesh, tree, 60.0, fb.FB_OP_A, prec, 0.5, 12))
            free.append(free_bytes())
        P = int(max(fb.fb_operator_info(ops[0])[2]))
        assert P == 43
        real, composed, phases = (P * (4 * P * P - 1) // 3 * 8, 32 * (4 * 32 * 32 - 1) // 3 * 16, (2 * P - 1) * 24)
        # the first operator on the tree alone pays for them; 316 M2L vectors and the octants' 16 at most
        kept = (free[0] - free[1]) - (free[1] - free[2])
        assert kept < 340 * (real + composed + phases)
        code = 5 * 49 + 4 * 7 + 3
        for n in (0, 7, 42):
            d64, d32 = (fb.fb_operator_export(op, 8, n, code).real for op in (ops[2], ops[0]))
            assert np.array_equal(d32, d64.astype(np.float32).astype(np.float64))
    finally:
        for op in ops:
            fb.fb_operator_destroy(op)
        fb.fb_tree_destroy(tree)
        fb.fb_mesh_destroy(mesh)
