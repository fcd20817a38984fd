"""Divergence and gradient of smooth fields, whose nodal values nearly cancel in every element, on shells of many
layers, where the radial differences are weighted with r = rho / (3 h): against the CPU FP64 oracle's geometry."""
import numpy as np
import pytest

from oracle import operators as O
from oracle.mesh import ShellMesh
from tests.layout import LayoutMap

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _fields(om, pm, a):
    x, y = om.node_xyz().T, pm.node_xyz().T
    u = np.stack([np.sin(2 * x[1] + a) + x[2] ** 2, np.cos(x[0] + x[2]) * (1 + a),
                  x[0] * x[1] * x[2] + 0.3 * np.sqrt((x * x).sum(0)) + a])
    return u, np.sin(2 * y[1] + a / 2) + y[2] ** 2


def _reference(om, pm, u, p):
    """B P u and P B^T p (free-slip) in 64 bits, element by element."""
    Pp, proj = O.prolongation(om, pm), O.boundary_projectors(om)
    pu, pf = O.project(proj, u), Pp @ p
    q, y = np.zeros(om.n_nodes), np.zeros((3, om.n_nodes))
    for ids in O._chunks(np.arange(om.n_wedges), 100000):
        nodes = om.wedge_nodes(ids)
        grad, V = O.wedge_geometry(om, ids)
        ue = pu[:, nodes]
        # differences to the wedge's mean value: the gradients of the six shape functions sum to zero
        div = np.einsum("dej,ejd->e", ue - ue.mean(axis=2, keepdims=True), grad)
        pc = pf[nodes].mean(axis=1)
        q += np.bincount(nodes.ravel(), weights=np.repeat(-V * div / 6, 6), minlength=om.n_nodes)
        for d in range(3):
            y[d] += np.bincount(nodes.ravel(), weights=(-(V * pc)[:, None] * grad[:, :, d]).ravel(), minlength=om.n_nodes)
    return Pp.T @ q, O.project(proj, y)


# Bounds in norm over the interior node layers: the errors of the form that takes the differences of nodal values
# first (radial sums and element contributions node by node), measured on these fields; the FP64 levels with
# N >= 32 run in double-float.  A form that rounds the layers' sums before their difference is at 1.1e-7 to 1.9e-7 (FP32,
# B) and 4.0e-14 (FP64, 101 layers, B).
@pytest.mark.parametrize("level,n_r,dtype,tol_b,tol_bt", [
    (3, 33, "f32", 7.1e-8, 3.1e-6), (4, 65, "f32", 7.0e-8, 6.1e-6), (5, 33, "f32", 8.8e-8, 3.4e-6),
    (5, 101, "f32", 8.1e-8, 8.3e-6), (5, 33, "f64", 2.9e-14, 2.6e-13), (5, 101, "f64", 3.1e-14, 8.4e-13)])
def test_smooth_fields(level, n_r, dtype, tol_b, tol_bt):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_21633_gb300 as tn
    td = torch.float64 if dtype == "f64" else torch.float32
    om = ShellMesh(level, n_r, 0.55, 1.0)
    pm = O.pressure_mesh(om)
    m = tn.tn_mesh_create(level, n_r, 0.55, 1.0)
    mp, pmap = LayoutMap(tn.tn_mesh_info(m, 0), om), LayoutMap(tn.tn_mesh_info(m, 1), pm)
    for a in (0.1, 1.0):
        u, p = _fields(om, pm, a)
        ud = [torch.tensor(mp.to_layout(v), device="cuda", dtype=td) for v in u]
        pd = torch.tensor(pmap.to_layout(p), device="cuda", dtype=td)
        q, y = torch.zeros_like(pd), [torch.zeros_like(t) for t in ud]
        tn.tn_apply_B(m, 0, ud, q)
        tn.tn_apply_BT(m, 0, pd, y)
        # the inputs as the library got them
        u = np.stack([mp.from_layout(t.double().cpu().numpy()) for t in ud])
        p = pmap.from_layout(pd.double().cpu().numpy())
        want_q, want_y = _reference(om, pm, u, p)
        for got, want, mesh, tol in ((pmap.from_layout(q.double().cpu().numpy())[None], want_q[None], pm, tol_b),
                                     (np.stack([mp.from_layout(t.double().cpu().numpy()) for t in y]), want_y, om, tol_bt)):
            k = np.arange(mesh.n_nodes) % mesh.n_r
            inside = (k > 0) & (k < mesh.n_r - 1)
            assert np.linalg.norm((got - want)[:, inside]) <= tol * np.linalg.norm(want[:, inside])
    tn.tn_mesh_destroy(m)
