"""Operators on levels with two node layers (the coarse level of a shell with three): both layers are boundary layers."""
import numpy as np
import pytest

from oracle import operators as O
from oracle.mesh import ShellMesh
from paper_2609_21633_gb300 import inputs
from tests.layout import LayoutMap, max_rel

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ORACLE_BC = {0: O.FREE, 1: O.NOSLIP}


# level 1 of a level-6 mesh has N = 32 (the smallest level of the tile-line kernels), of a level-5 mesh N = 16
@pytest.mark.parametrize("level,kappa,quad,bc", [(6, 0.0, 1, (0, 0)), (6, 0.3, 1, (0, 0)), (6, 0.0, 1, (1, 0)),
                                                 (6, 0.0, 2, (0, 0)), (5, 0.3, 1, (0, 1))])
def test_apply_and_diag(level, kappa, quad, bc):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_21633_gb300 as tn
    om = ShellMesh(level - 1, 2, 0.55, 1.0)
    P = O.boundary_projectors(om, (ORACLE_BC[bc[0]], ORACLE_BC[bc[1]]))
    m = tn.tn_mesh_create(level, 3, 0.55, 1.0, bc[0], bc[1], hg_kappa=kappa, radial_quad_points=quad)
    info = tn.tn_mesh_info(m, 1)
    mp = LayoutMap(info, om)
    fine = torch.tensor(inputs.lognormal_viscosity(tn.tn_mesh_info(m, 0)["n_wedges"], 4), device="cuda")
    tn.tn_set_viscosity(m, fine)
    eta1 = torch.zeros(info["n_wedges"], device="cuda", dtype=torch.float64)
    tn.tn_get_viscosity(m, 1, eta1)
    eta = mp.wedges_from_layout(eta1.cpu().numpy())
    u = inputs.normal((3, om.n_nodes), 5)
    want_y = O.apply_A_constrained(om, eta, u, P, kappa=kappa, quad=quad)
    want_d = O.diag_A_constrained(om, eta, P, kappa=kappa, quad=quad)
    for dtype, tol in ((torch.float64, 1e-12), (torch.float32, 1e-5)):  # 1e-12 is the FP64 bar of the operator tests, 1e-5 half the FP32 one
        ud = [torch.tensor(mp.to_layout(v), device="cuda", dtype=dtype) for v in u]
        y, d = [torch.zeros_like(t) for t in ud], [torch.zeros_like(t) for t in ud]
        tn.tn_apply_A(m, 1, ud, y)
        tn.tn_diag_A(m, 1, d)
        assert max_rel(np.stack([mp.from_layout(t.double().cpu().numpy()) for t in y]), want_y) <= tol
        assert max_rel(np.stack([mp.from_layout(t.double().cpu().numpy()) for t in d]), want_d) <= tol
    tn.tn_mesh_destroy(m)
