"""Divergence and gradient with the pressure transfers inside one kernel, against the CPU FP64 oracle: the
smallest tiles, levels with strips of more than one CTA's nodes, more coarse layers than one radial chunk holds,
unaligned FP32 vectors."""
import numpy as np
import pytest

from oracle import operators as O
from oracle.mesh import ShellMesh
from paper_2609_21633_gb300 import inputs
from tests.layout import LayoutMap, max_rel

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ORACLE_BC = {0: O.FREE, 1: O.NOSLIP}


@pytest.mark.parametrize("level,n_r,bc", [(2, 3, (0, 0)), (2, 131, (1, 0)), (3, 9, (0, 1)), (4, 5, (0, 0)), (5, 7, (1, 1)),
                                          (5, 11, (0, 0)), (6, 3, (0, 0))])
@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_div_grad(level, n_r, bc, dtype):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_21633_gb300 as tn
    td = torch.float64 if dtype == "f64" else torch.float32
    om = ShellMesh(level, n_r, 0.55, 1.0)
    pm = O.pressure_mesh(om)
    m = tn.tn_mesh_create(level, n_r, 0.55, 1.0, bc[0], bc[1])
    info, pinfo = tn.tn_mesh_info(m, 0), tn.tn_mesh_info(m, 1)
    mp, pmap = LayoutMap(info, om), LayoutMap(pinfo, pm)
    B = O.assemble_B(om, O.prolongation(om, pm))
    Pm = O.projector_matrix(O.boundary_projectors(om, (ORACLE_BC[bc[0]], ORACLE_BC[bc[1]])))

    def buf(n, vals=None):  # one element past an allocation's start
        t = torch.zeros(n + 1, device="cuda", dtype=td)[1:]
        if vals is not None:
            t.copy_(torch.tensor(vals, device="cuda"))
        return t

    u = inputs.normal((3, om.n_nodes), 11)
    p = inputs.normal(pm.n_nodes, 12)
    ud = [buf(info["n_layout"], mp.to_layout(u[c])) for c in range(3)]
    pd = buf(pinfo["n_layout"], pmap.to_layout(p))
    q, y = buf(pinfo["n_layout"]), [buf(info["n_layout"]) for _ in range(3)]
    tn.tn_apply_B(m, 0, ud, q)
    tn.tn_apply_BT(m, 0, pd, y)
    tol = 1e-12 if dtype == "f64" else 2e-5
    assert max_rel(pmap.from_layout(q.double().cpu().numpy()), B @ (Pm @ u.ravel())) <= tol
    want = (Pm @ (B.T @ p)).reshape(3, -1)
    assert max_rel(np.stack([mp.from_layout(t.double().cpu().numpy()) for t in y]), want) <= tol
    q2, y2 = buf(pinfo["n_layout"]), [buf(info["n_layout"]) for _ in range(3)]
    tn.tn_apply_B(m, 0, ud, q2)
    tn.tn_apply_BT(m, 0, pd, y2)
    assert torch.equal(q, q2) and all(torch.equal(a, b) for a, b in zip(y, y2))
    tn.tn_mesh_destroy(m)
