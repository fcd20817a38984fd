"""The double-float A apply (FP64 levels with N >= 32) against the CPU FP64 oracle at the edges of its
range: one cell-layer chunks, odd layer counts, the smallest shell, smooth inputs whose element
differences cancel."""
import numpy as np
import pytest

from oracle import operators as O
from oracle.mesh import ShellMesh
from paper_2609_21633_gb300 import inputs
from tests.layout import LayoutMap, max_rel

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ORACLE_BC = {0: O.FREE, 1: O.NOSLIP}


@pytest.mark.parametrize("n_r,bc,kappa,div_term,smooth", [
    (3, (0, 0), 0.0, True, False), (3, (1, 1), 0.3, True, False), (7, (1, 0), 0.3, False, False),
    (13, (0, 1), 0.0, False, False), (19, (0, 0), 0.0, True, True), (11, (0, 0), 0.3, True, True)])
def test_apply_A_double_float(n_r, bc, kappa, div_term, smooth):
    """Bar 1e-12 of the largest value.  Smooth fields: the result is about h^2 of the summands, so the bar is
    taken of the largest element contribution, eta |u| / h, through the largest diagonal entry."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_21633_gb300 as tn
    om = ShellMesh(5, n_r, 0.55, 1.0)
    P = O.boundary_projectors(om, (ORACLE_BC[bc[0]], ORACLE_BC[bc[1]]))
    eta = inputs.lognormal_viscosity(om.n_wedges, 3) if not smooth else np.ones(om.n_wedges)
    m = tn.tn_mesh_create(5, n_r, 0.55, 1.0, bc[0], bc[1], div_term, hg_kappa=kappa)
    mp = LayoutMap(tn.tn_mesh_info(m, 0), om)
    tn.tn_set_viscosity(m, torch.tensor(mp.wedges_to_layout(eta), device="cuda"))
    if smooth:
        x = om.node_xyz().T
        u = np.stack([np.sin(2 * x[1]) + x[2] ** 2, np.cos(x[0] + x[2]), x[0] * x[1] * x[2]])
    else:
        u = inputs.normal((3, om.n_nodes), 10)
    want = O.apply_A_constrained(om, eta, u, P, div_term=div_term, kappa=kappa)
    ud = [torch.tensor(mp.to_layout(u[c]), device="cuda") for c in range(3)]
    y = [torch.zeros_like(t) for t in ud]
    tn.tn_apply_A(m, 0, ud, y)
    got = np.stack([mp.from_layout(t.cpu().numpy()) for t in y])
    scale = np.abs(want).max()
    if smooth:
        scale = np.abs(u).max() * np.abs(O.diag_A_constrained(om, eta, P, div_term=div_term, kappa=kappa)).max()
    assert np.abs(got - want).max() <= 1e-12 * scale
    y2 = [torch.zeros_like(t) for t in ud]
    tn.tn_apply_A(m, 0, ud, y2)
    assert all(torch.equal(a, b) for a, b in zip(y, y2))
    tn.tn_mesh_destroy(m)
