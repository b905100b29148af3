"""Receiver evaluation split over the CTAs of a cluster: receiver counts on
both sides of the rule's lines (1 to 8 shares), receivers near a wall
(closed-form entries) and far from it, against the oracle's direct sum in
FP64 (3-point rule and closed forms; 1e-11 covers the rounding of sums of a
few thousand terms with phases to k R ~ 60)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2103_16073_gb300 as fb
from _cases import oracle_mesh, rel, seeded_vector, workload
from oracle import bem


@pytest.mark.parametrize("name", ["ragged", "sub"])
@pytest.mark.parametrize("nrec", [1, 7, 150, 1000])
def test_field_matches_oracle(name, nrec):
    wl = workload(name)
    rng = np.random.default_rng(nrec)
    rec = np.array(wl.room) * rng.uniform(0.001, 0.999, size=(nrec, 3))
    psi, gam = seeded_vector(wl.n, 1), seeded_vector(wl.n, 2)
    src = np.array(wl.room) * 0.4
    mesh = fb.fb_mesh_create(wl.verts, wl.tris)
    fb.fb_mesh_set_admittance(mesh, wl.beta)
    try:
        out = torch.empty(nrec, dtype=torch.complex128, device="cuda")
        args = [torch.tensor(a, device="cuda") for a in (psi, gam, rec)]
        got = fb.fb_eval_field(mesh, wl.k, *args, out, src=src).cpu().numpy()
    finally:
        fb.fb_mesh_destroy(mesh)
    pick = np.linspace(0, nrec - 1, min(nrec, 40)).astype(int)
    want = bem.receiver_field(oracle_mesh(name), wl.k, wl.beta, psi, gam, rec[pick], src)
    assert rel(got[pick], want) < 1e-11
